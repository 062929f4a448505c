"""Launches of few particles (three lanes each) and of many (one lane each)
give every particle the same result, bit for bit, in FP64 and in mixed
precision: the same particles alone and repeated beyond the limit, over every
option, at sizes around a warp's ten particles, in batches too."""
import numpy as np
import pytest

from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu

# particles of a launch up to which each has three lanes
LIMIT = {mp.PREC_FP64: 18240, mp.PREC_MIXED: 30400}


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = mp.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def fields():
    wells = I.random_box_field(5, 19, 23, seed=61, lnk_var=2.5, n_wells=6, n_inactive=9, well_scale=4.0)
    flat = I.cfg1_field()                                                  # one layer: an axis without flow
    return {"wells": wells, "flat": flat}


def _run(ctx, fh, cells, frac, t0, times, kw):
    g = ctx.release_explicit(fh, cells, frac, t0)
    req = ctx.track(g, times=times, **kw)
    ep = req.endpoints()
    ts = req.timeseries() if req.n_times else None
    pl = req.pathlines() if kw["mode"] & mp.MODE_PATHLINE else None
    st = req.stats()
    if pl is not None:
        pl = pl[np.lexsort((pl["seq"], pl["particle"]))]
    if kw.get("flags", 0) & mp.TRACK_UPDATE_GROUP:   # go on from the stop time
        more = ctx.track(g, **{**kw, "mode": mp.MODE_ENDPOINT, "t_stop": np.inf})
        ep = {**ep, **{"then_" + k: v for k, v in more.endpoints().items()}}
        more.free()
    req.free()
    mp.mp_group_free(g)
    return ep, ts, pl, st


@pytest.mark.parametrize("precision", [mp.PREC_FP64, mp.PREC_MIXED])
@pytest.mark.parametrize("name", ["wells", "flat"])
@pytest.mark.parametrize("n", [1, 9, 10, 11, 257])
@pytest.mark.parametrize("option", ["endpoint", "times", "paths", "all", "weak sinks", "stop and resume", "step cap"])
def test_few_equal_many(ctx, fields, precision, name, n, option):
    f = fields[name]
    fh = ctx.field(f)
    rng = np.random.default_rng(n)
    cells, frac = I.explicit_particles(f, n, seed=n, active_only=(option != "all"))
    frac[rng.random(n) < 0.2] = rng.integers(0, 2, 3)      # some on corners
    ta = I.t_adv_of(f, 1e-4, 0.3)
    t0 = rng.random(n) * 0.2 * ta if option in ("all", "times") else None
    times = I.log_times(ta, 13) if option in ("times", "all", "weak sinks", "step cap") else None
    kw = {"mode": mp.MODE_ENDPOINT | (mp.MODE_TIMESERIES if times is not None else 0), "precision": precision}
    if option in ("paths", "all"):
        kw.update(mode=kw["mode"] | mp.MODE_PATHLINE, path_capacity=3000000)
    if option == "weak sinks":
        kw.update(flags=mp.TRACK_PASS_WEAK_SINKS, weak_sink_fraction=0.4)
    if option == "stop and resume":
        kw.update(flags=mp.TRACK_UPDATE_GROUP, t_stop=0.1 * ta)
    if option == "step cap":
        kw.update(max_steps=7)
    few = _run(ctx, fh, cells, frac, t0, times, kw)
    rep = LIMIT[precision] // n + 1
    many = _run(ctx, fh, np.tile(cells, rep), np.tile(frac, (rep, 1)), None if t0 is None else np.tile(t0, rep), times, kw)
    assert many[0]["t"].size > LIMIT[precision] >= n
    for k, v in few[0].items():
        w = many[0][k].reshape(rep, n)
        assert (w.view(np.uint8) == np.ascontiguousarray(v).view(np.uint8).reshape(-1)).all(), k
    if times is not None:
        w = np.ascontiguousarray(many[1].reshape(len(times), rep, n)[:, [0, rep - 1]]).view(np.uint8)
        v = np.ascontiguousarray(np.repeat(few[1][:, None], 2, 1)).view(np.uint8)
        assert np.array_equal(w, v)
    if few[2] is not None and many[3]["path_points"] <= 3000000:
        first = many[2][many[2]["particle"] < n]
        assert np.array_equal(first.view(np.uint8), few[2].view(np.uint8))
    assert many[3]["n_status"] == [rep * v for v in few[3]["n_status"]]
    assert many[3]["cell_steps"] == rep * few[3]["cell_steps"]
    assert few[3]["device_error"] == 0
    mp.mp_field_free(fh)


@pytest.mark.parametrize("precision", [mp.PREC_FP64, mp.PREC_MIXED])
def test_batch_of_few_equals_alone_among_many(ctx, fields, precision):
    f = fields["wells"]
    fh = ctx.field(f)
    times = I.log_times(I.t_adv_of(f, 1e-4, 0.3), 9)
    opts = [mp.make_opts(mode=mp.MODE_ENDPOINT | (mp.MODE_TIMESERIES if i % 2 else 0), times=times if i % 2 else None,
                         precision=precision) for i in range(12)]
    parts = [I.explicit_particles(f, 7 + 11 * i, seed=90 + i) for i in range(12)]

    def batch(extra):
        groups = [ctx.release_explicit(fh, c, x) for c, x in parts]
        more = [ctx.release_explicit(fh, *I.explicit_particles(f, extra, seed=3))] if extra else []
        ids = mp.mp_track_batch(ctx.h, groups + more, opts + [mp.make_opts(precision=precision)] * len(more))
        out = []
        for i, (r, (c, _)) in enumerate(zip(ids, parts)):
            out.append(mp.mp_get_endpoints(ctx.h, r, c.size))
            if i % 2:
                out[-1]["ts"] = mp.mp_get_timeseries(ctx.h, r, c.size, 9).view(np.uint8)
        for r in ids:
            mp.mp_req_free(ctx.h, r)
        for g in groups + more:
            mp.mp_group_free(g)
        return out

    for a, b in zip(batch(0), batch(LIMIT[precision] + 1)):
        for k in a:
            assert np.array_equal(np.ascontiguousarray(a[k]).view(np.uint8), np.ascontiguousarray(b[k]).view(np.uint8)), k
    mp.mp_field_free(fh)
