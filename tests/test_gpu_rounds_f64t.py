"""The mixed form with FP64 time gives every particle its result whatever the
launch's shape: particle counts around its rounds of at most 16 warps an SM,
blocks and fetches chosen and given, against the static schedule, bit for
bit."""
import numpy as np
import pytest

from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 5000, 77824, 77825, 155649])
@pytest.mark.parametrize("mode", [mp.MODE_ENDPOINT, mp.MODE_ENDPOINT | mp.MODE_TIMESERIES,
                                  mp.MODE_ENDPOINT | mp.MODE_TIMESERIES | mp.MODE_PATHLINE])
def test_persistent_equals_static(n, mode):
    w = I.workload("cfg1")
    kw = {"mode": mode, "precision": mp.PREC_MIXED_F64T, "path_capacity": 200 * n,
          "times": w.times[::10] if mode & mp.MODE_TIMESERIES else None}
    with mp.Context(0) as ctx:
        fh = ctx.field(w.field)
        gh = ctx.release_box(fh, n, w.release.lo, w.release.hi, 5)
        outs = []
        for more in ({"schedule": mp.SCHED_STATIC}, {}, {"block": 96}, {"block": 256, "steps_per_fetch": 1}):
            req = ctx.track(gh, **kw, **more)
            ep, st = req.endpoints(), req.stats()
            out = {k: v.view(np.uint8) for k, v in ep.items()}
            if mode & mp.MODE_TIMESERIES:
                out["ts"] = req.timeseries().view(np.uint8)
            if mode & mp.MODE_PATHLINE:
                assert st["path_points"] <= 200 * n
                pl = req.pathlines()
                out["path"] = pl[np.lexsort((pl["seq"], pl["particle"]))].view(np.uint8)
            outs.append((out, st["n_status"], st["cell_steps"]))
            req.free()
        for got in outs[1:]:
            for k in outs[0][0]:
                assert np.array_equal(got[0][k], outs[0][0][k]), k
            assert got[1:] == outs[0][1:]
        mp.mp_group_free(gh)
