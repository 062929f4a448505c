"""The persistent schedule gives every particle its result whatever the
launch's shape: particle counts around what fits on the GPU at once (one
round, the first of two, of three), block sizes chosen and given, against the
static schedule, bit for bit."""
import numpy as np
import pytest

from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = mp.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n", [18241, 77824, 77825, 97281, 155649, 233473])
@pytest.mark.parametrize("times", [0, 5])
def test_persistent_equals_static(ctx, n, times):
    w = I.workload("cfg1")
    fh = ctx.field(w.field)
    kw = {"mode": mp.MODE_ENDPOINT | (mp.MODE_TIMESERIES if times else 0), "times": w.times[::10] if times else None}
    gh = ctx.release_box(fh, n, w.release.lo, w.release.hi, 5)
    outs = []
    for more in ({"schedule": mp.SCHED_STATIC}, {}, {"block": 96}, {"block": 256, "steps_per_fetch": 1}):
        req = ctx.track(gh, **kw, **more)
        ep, st = req.endpoints(), req.stats()
        outs.append(({k: v.view(np.uint8) for k, v in ep.items()}, req.timeseries().view(np.uint8) if times else None, st))
        req.free()
    for ep, ts, st in outs[1:]:
        for k in ep:
            assert np.array_equal(ep[k], outs[0][0][k]), k
        assert ts is None or np.array_equal(ts, outs[0][1])
        assert st["n_status"] == outs[0][2]["n_status"] and st["cell_steps"] == outs[0][2]["cell_steps"]
    mp.mp_group_free(gh)
    mp.mp_field_free(fh)
