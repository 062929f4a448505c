"""The static and the persistent one-lane kernels on launches too large for
three lanes a particle, over every option and in batches: the same particles
repeated beyond that limit, FP64 against the oracle, both precisions against
the launch of the particles alone, every copy bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

LIMIT = {mp.PREC_FP64: 18240, mp.PREC_MIXED: 30400}   # on 152 multiprocessors
N = 1300
PASS = mp.TRACK_PASS_WEAK_SINKS
SHAPES = [(mp.SCHED_STATIC, 0), (mp.SCHED_STATIC, 96), (mp.SCHED_DYNAMIC, 0), (mp.SCHED_DYNAMIC, 128)]
OPTIONS = ["plain", "times", "paths", "pass sinks", "threshold", "resume", "step cap", "staged", "periods"]


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = mp.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def model(ctx):
    f = I.random_box_field(4, 17, 21, seed=40, lnk_var=1.5, n_wells=6, n_inactive=7, well_scale=8.0)
    fs = I.period_fields(f, seed=6, head_scale=(1.0, 0.4, -0.7), new_wells=(0, 2, 1), well_scale=3.0)
    cells, frac = I.explicit_particles(f, N, seed=12, cols=(1, 6))
    st0 = O.release_explicit(f, cells, frac)
    full = O.track(f, st0, pass_weak_sinks=True, arith="mirror")
    fhs = [ctx.field(g) for g in fs]
    yield f, fs, fhs, cells, frac.reshape(N, 3), st0, full
    for fh in fhs:
        mp.mp_field_free(fh)


def _case(model, option):
    """Track options, release times, and the oracle's results of a case."""
    f, fs, fhs, cells, frac, st0, full = model
    t = np.quantile(full["t"], [0.1, 0.3, 0.5, 0.9])
    kw, ok, t0 = {"mode": mp.MODE_ENDPOINT}, {}, None
    if option in ("times", "paths", "pass sinks", "threshold", "step cap", "periods", "staged"):
        kw.update(mode=mp.MODE_ENDPOINT | mp.MODE_TIMESERIES, times=np.sort(np.append(t, [t[1], 2 * t[3]])))
    if option == "paths":
        kw.update(mode=kw["mode"] | mp.MODE_PATHLINE)
        ok.update(pathline=True)
    if option in ("pass sinks", "threshold", "resume", "periods"):
        kw.update(flags=PASS)
        ok.update(pass_weak_sinks=True)
    if option == "threshold":
        kw.update(weak_sink_fraction=0.6)
        ok.update(weak_sink_fraction=0.6)
    if option == "step cap":
        kw.update(max_steps=6)
        ok.update(max_steps=6)
    state = dict(st0)
    if option == "staged":
        t0 = np.where(np.arange(N) % 3 == 0, 0.4 * t[2], 0.0)
        state["t"] = t0
        kw.update(t_stop=t[2])
        ok.update(t_stop=t[2])
    times = kw.get("times")
    if option == "resume":
        kw.update(flags=PASS | mp.TRACK_UPDATE_GROUP, t_stop=t[1])
        first = O.track(f, state, t_stop=t[1], arith="mirror", **ok)
        ref = [first, O.track(f, O.resume_state(first), arith="mirror", **ok)]
    elif option == "periods":
        ref = [O.track_periods(fs, [t[1], t[2]], state, times=times, arith="mirror", **ok)]
    else:
        ref = [O.track(f, state, times=times, arith="mirror", **ok)]
    return kw, t0, ref, [t[1], t[2]]


def _run(ctx, model, option, kw, t0, ends, precision, rep, **shape):
    f, fs, fhs, cells, frac, st0, full = model
    n = N * rep
    g = ctx.release_explicit(fhs[0], np.tile(cells, rep), np.tile(frac, (rep, 1)), None if t0 is None else np.tile(t0, rep))
    kw = dict(kw, precision=precision, path_capacity=400 * n, **shape)
    req = ctx.track_periods(g, fhs, ends, **kw) if option == "periods" else ctx.track(g, **kw)
    out = [req.endpoints()]
    ts = req.timeseries() if req.n_times else None
    path = None
    if kw["mode"] & mp.MODE_PATHLINE:
        assert req.stats()["path_points"] <= 400 * n
        path = np.sort(req.pathlines(), order=["particle", "seq"])
    assert req.stats()["device_error"] == 0
    req.free()
    if option == "resume":
        more = ctx.track(g, **{**kw, "t_stop": np.inf})
        out.append(more.endpoints())
        more.free()
    mp.mp_group_free(g)
    return out, ts, path


@pytest.mark.parametrize("precision", [mp.PREC_FP64, mp.PREC_MIXED])
@pytest.mark.parametrize("option", OPTIONS)
def test_schedules_beyond_the_limit(ctx, model, precision, option):
    f = model[0]
    kw, t0, ref, ends = _case(model, option)
    rep = LIMIT[precision] // N + 1
    few = _run(ctx, model, option, kw, t0, ends, precision, 1)
    for schedule, block in SHAPES:
        out, ts, path = _run(ctx, model, option, kw, t0, ends, precision, rep, schedule=schedule, block=block)
        for got, alone, want in zip(out, few[0], ref):
            if precision == mp.PREC_FP64:
                G.compare_fp64({k: v[:N] for k, v in got.items()}, want, dmin=G.dmin(f))
            for k, v in alone.items():
                assert (got[k].reshape(rep, N).view(np.uint8) == v.view(np.uint8)).all(), (k, schedule, block)
        if ts is not None:
            if precision == mp.PREC_FP64:
                G.compare_timeseries_fp64(np.ascontiguousarray(ts[:, :N]), ref[0], dmin=G.dmin(f))
            whole = ts.reshape(len(kw["times"]), rep, N)
            for c in (0, rep // 2, rep - 1):
                assert np.array_equal(np.ascontiguousarray(whole[:, c]).view(np.uint8), few[1].view(np.uint8)), (schedule, block)
        if path is not None:
            for c in (0, rep - 1):
                mine = path[(path["particle"] >= c * N) & (path["particle"] < (c + 1) * N)].copy()
                mine["particle"] -= c * N
                assert np.array_equal(mine.view(np.uint8), few[2].view(np.uint8)), (schedule, block)


@pytest.mark.parametrize("precision", [mp.PREC_FP64, mp.PREC_MIXED])
@pytest.mark.parametrize("schedule,block", SHAPES)
def test_batch_beyond_the_limit(ctx, model, precision, schedule, block):
    f, fs, fhs, cells, frac, st0, full = model
    times = np.quantile(full["t"], [0.1, 0.5, 0.9])
    sizes = [1, 31, 700, 0, 5000, 12000, 20000]           # 37,732 in one launch
    kws = [{"mode": mp.MODE_ENDPOINT | (mp.MODE_TIMESERIES if i % 2 else 0), "times": times if i % 2 else None,
            "flags": PASS if i % 3 == 0 else 0, "precision": precision, "max_steps": 9 if i == 4 else 0}
           for i in range(len(sizes))]
    take = [(np.arange(m) + 17 * i) % N for i, m in enumerate(sizes)]
    groups = [ctx.release_explicit(fhs[0], cells[t], frac[t]) for t in take]
    ids = mp.mp_track_batch(ctx.h, groups, [mp.make_opts(schedule=schedule, block=block, **kw) for kw in kws])
    for i, (r, t, kw, g) in enumerate(zip(ids, take, kws, groups)):
        if t.size:
            alone = ctx.release_explicit(fhs[0], cells, frac)
            req = ctx.track(alone, **kw)
            ep, ts = req.endpoints(), req.timeseries() if req.n_times else None
            got = mp.mp_get_endpoints(ctx.h, r, t.size)
            for k, v in ep.items():
                assert np.array_equal(got[k].view(np.uint8), np.ascontiguousarray(v[t]).view(np.uint8)), (k, i)
            if ts is not None:
                rec = mp.mp_get_timeseries(ctx.h, r, t.size, len(times))
                assert np.array_equal(rec.view(np.uint8), np.ascontiguousarray(ts[:, t]).view(np.uint8)), i
            req.free()
            mp.mp_group_free(alone)
        mp.mp_req_free(ctx.h, r)
        mp.mp_group_free(g)
