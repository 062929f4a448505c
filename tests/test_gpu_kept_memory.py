"""Device memory that a context keeps from freed fields is given back when an
allocation of the context would otherwise fail."""
import pytest

from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sync", [False, True])
def test_kept_memory_is_given_back_when_short(sync):
    import torch
    f = I.random_box_field(20, 200, 200, seed=3, lnk_var=0.5)
    with mp.Context(0) as ctx:
        small = ctx.field(I.random_box_field(3, 9, 11, seed=1, lnk_var=0.5))
        fh = ctx.field(f)
        held = mp.mp_field_bytes(fh)
        assert held > 100 << 20
        mp.mp_field_free(fh)
        if sync:
            torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        cells, frac = I.explicit_particles(I.random_box_field(3, 9, 11, seed=1, lnk_var=0.5), 10, seed=2)
        gh = ctx.release_explicit(small, cells, frac)
        with pytest.raises(mp.MPError) as e:              # (an allocation that no GPU can give)
            ctx.track(gh, mode=mp.MODE_ENDPOINT | mp.MODE_PATHLINE, path_capacity=1 << 44)
        assert e.value.code == -4
        assert torch.cuda.mem_get_info()[0] - before >= held - (32 << 20)
        r = ctx.track(gh)
        assert r.stats()["device_error"] == 0
        r.free()
        mp.mp_group_free(gh)
