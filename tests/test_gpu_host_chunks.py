"""mp_track_host gives the same results however many chunks it launches ahead
of the one it reads: counts around that number, uneven last chunks, host arrays
pinned and pageable, against one chunk, bit for bit."""
import numpy as np
import pytest

from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("precision", [mp.PREC_FP64, mp.PREC_MIXED])
def test_chunks_equal_one(precision, pinned):
    import torch
    f = I.random_box_field(5, 19, 23, seed=17, lnk_var=2.0, n_wells=5, n_inactive=9)
    n, nt = 10007, 6
    cells, frac = I.explicit_particles(f, n, seed=2)
    opts = mp.make_opts(mode=mp.MODE_ENDPOINT | mp.MODE_TIMESERIES, precision=precision,
                        times=I.log_times(I.t_adv_of(f, 1e-4, 0.3), nt))

    def array(m, d):
        size = m * np.dtype(d).itemsize
        return torch.empty(size, dtype=torch.uint8, pin_memory=pinned).numpy().view(d)

    with mp.Context(0) as ctx:
        fh = ctx.field(f)
        ref = mp.mp_track_host(ctx.h, fh, cells, frac, opts, n_chunks=1)
        for chunks in (2, 3, 4, 5, 7, 16, 1000):
            out = {k: array(n, d) for k, d in mp.ENDPOINT_DTYPES.items()}
            ts = array(nt * n, mp.TS_RECORD).reshape(nt, n)
            _, _, st = mp.mp_track_host(ctx.h, fh, cells, frac, opts, n_chunks=chunks, out=out, ts_out=ts)
            for k in out:
                assert np.array_equal(out[k].view(np.uint8), ref[0][k].view(np.uint8)), (k, chunks)
            assert np.array_equal(ts.view(np.uint8), ref[1].view(np.uint8)), chunks
            assert st["n_status"] == ref[2]["n_status"] and st["cell_steps"] == ref[2]["cell_steps"]
        # a chunk that cannot be launched, ahead or later: its error, and nothing left running
        for bad in (5, n // 2, n - 1):
            wrong = frac.reshape(-1, 3).copy()
            wrong[bad] = np.nan
            with pytest.raises(mp.MPError) as e:
                mp.mp_track_host(ctx.h, fh, cells, wrong, opts, n_chunks=7)
            assert e.value.code == -3
        again = mp.mp_track_host(ctx.h, fh, cells, frac, opts, n_chunks=7)
        assert np.array_equal(again[1].view(np.uint8), ref[1].view(np.uint8))
