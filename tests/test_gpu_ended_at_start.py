"""Particles whose track ends before its first step (a release in an inactive
cell, at or after the stop time) are written out with the others of their warp:
whole warps of them and single ones, in both schedules and with several steps
a fetch, against launches of few particles, bit for bit."""
import numpy as np
import pytest

from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu

N, PART = 40007, 10000   # (a part is tracked by the form for few particles)


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = mp.Context(0)
    yield c
    c.close()


def _track(ctx, fh, cells, frac, t0, **kw):
    g = ctx.release_explicit(fh, cells, frac, t0)
    req = ctx.track(g, mode=mp.MODE_ENDPOINT | mp.MODE_TIMESERIES | mp.MODE_PATHLINE, **kw)
    ep, ts, st, pl = req.endpoints(), req.timeseries(), req.stats(), req.pathlines()
    req.free()
    mp.mp_group_free(g)
    return ep, ts, st, np.sort(pl, order=("particle", "seq"))


@pytest.mark.parametrize("precision", [mp.PREC_FP64, mp.PREC_MIXED])
def test_ended_at_start(ctx, precision):
    f = I.random_box_field(5, 19, 23, seed=67, lnk_var=2.0, n_wells=5, n_inactive=40, well_scale=4.0)
    fh = ctx.field(f)
    cells, frac = I.explicit_particles(f, N, seed=9, active_only=False)
    i = np.arange(N)
    ta = I.t_adv_of(f, 1e-4, 0.3)
    stop = 0.5 * ta
    t0 = np.where((i % 640 < 128) | (i % 37 == 0) | (i >= N - 70), stop * (1 + i % 2), 0.0)   # whole warps, single lanes, the last ones
    kw = {"times": np.linspace(0.02, 0.6, 9) * ta, "t_stop": stop, "precision": precision, "max_steps": 500,
          "path_capacity": 4000000}
    parts = [_track(ctx, fh, cells[a:a + PART], frac[a:a + PART], t0[a:a + PART], **kw) for a in range(0, N, PART)]
    ep = {k: np.concatenate([p[0][k] for p in parts]) for k in parts[0][0]}
    ts = np.concatenate([p[1] for p in parts], axis=1)
    assert (ep["steps"] == 0).sum() > N // 5 and (ep["steps"] > 0).any()
    for more in ({}, {"steps_per_fetch": 1}, {"steps_per_fetch": 16, "block": 128}, {"schedule": mp.SCHED_STATIC}):
        e, t, st, pl = _track(ctx, fh, cells, frac, t0, **kw, **more)
        for k in ep:
            assert np.array_equal(e[k].view(np.uint8), ep[k].view(np.uint8)), (k, more)
        assert np.array_equal(t.view(np.uint8), ts.view(np.uint8)), more
        assert list(st["n_status"]) == [sum(p[2]["n_status"][j] for p in parts) for j in range(len(st["n_status"]))]
        assert st["cell_steps"] == sum(p[2]["cell_steps"] for p in parts)
        for a, p in zip(range(0, N, PART), parts):
            mine = pl[(pl["particle"] >= a) & (pl["particle"] < a + PART)].copy()
            mine["particle"] -= a
            assert np.array_equal(mine.view(np.uint8), p[3].view(np.uint8)), more
    mp.mp_field_free(fh)
