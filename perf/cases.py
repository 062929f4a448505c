"""Timed cases of the particle tracker: what a user's program has it do, through
the Python binding of libmp.

Every case is one call sequence of a user's program: release particles on a
loaded flow field, track them, read the results, free the handles.  The flow
fields are lognormal aquifers (exponential covariance, constant heads west and
east at unit mean gradient, pumping wells) made on the GPU from the seed, of
the sizes of this repository's workloads and tests.

Kinds (the "kind" of a case):
  track     one request on a rectilinear field; results read into device tensors
  paths     the same with pathlines from a staged explicit release, the points
            put in (particle, step) order as a plot or a file needs them
  periods   piecewise-steady flow: three stress periods, weak sinks passed
  batch     many uneven requests in one launch, as a server admits them
  host      host arrays in, host arrays out (mp_track_host)
  coupled   a flow model's time step: load its new face flows from device
            arrays, track the particles on through them, drop the field
  quadtree  one request on a quadtree grid
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2302_13590_gb300 import mp
from paper_2302_13590_gb300.inputs import usg

KINDS = ("track", "track", "track", "paths", "periods", "batch", "host", "coupled", "quadtree")
FP64, MIXED = "fp64", "mixed"
LNK_MEAN = -9.2   # mean of ln K (m/s)
POROSITY = 0.3
INF = math.inf


def _case(name, kind, shape, n, precision, times=0, var=1.0, wells=0, uniform=True, reqs=1):
    c = {"name": name, "kind": kind, "nlay": shape[0], "nrow": shape[1], "ncol": shape[2], "n": n,
         "precision": precision, "times": times, "var": var, "wells": wells, "uniform": uniform, "reqs": reqs}
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # a first model: one homogeneous layer with a pumping well, 1000 particles, endpoints (a call's latency)
        _case("one_layer_1k", "track", (1, 50, 50), 1000, FP64, var=0.0, wells=1),
        # a served request of usual size: mixed precision, endpoints and 20 output times
        _case("served_request_4k", "track", (20, 200, 200), 4000, MIXED, times=20),
        # a capture-zone study: endpoints of 30,000 particles through a 3-D heterogeneous aquifer
        _case("capture_zone_30k", "track", (20, 200, 200), 30000, FP64),
        # the benchmark workload: a million particles, endpoints and 50 output times, double precision
        _case("breakthrough_fp64_1m", "track", (20, 200, 200), 1000000, FP64, times=50),
        # the same in mixed precision
        _case("breakthrough_mixed_1m", "track", (20, 200, 200), 1000000, MIXED, times=50),
        # a large, heterogeneous well field of varying porosity in mixed precision, 20 output times
        _case("well_field_mixed_2m", "track", (40, 400, 400), 2000000, MIXED, times=20, var=1.5, wells=20),
        # pathlines for plotting, odd sizes, irregular spacing, a staged release
        _case("pathlines_ragged", "paths", (7, 61, 83), 5003, FP64, wells=3, uniform=False),
        # three stress periods, weak wells passed through, 20 output times
        _case("stress_periods_50k", "periods", (10, 100, 120), 50000, FP64, times=20, wells=4),
        # a server's admission pass: 24 uneven requests in one launch
        _case("admitted_batch_24", "batch", (20, 200, 200), 240000, MIXED, times=20, reqs=24),
        # a host program's call: numpy arrays in and out
        _case("host_to_host_200k", "host", (20, 200, 200), 200000, FP64, times=10),
        # one time step of a coupled transient flow model: new face flows, 10,000 particles on through them
        _case("coupled_step_10k", "coupled", (20, 200, 200), 10000, FP64),
        # a quadtree refinement around wells
        _case("quadtree_100k", "quadtree", (6, 36, 40), 100000, FP64, times=10, wells=3),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(KINDS)
    precision = FP64 if kind in ("quadtree", "coupled") else rng.choice((FP64, FP64, MIXED))
    wells = rng.randint(0, 6)
    var = rng.choice((0.5, 1.0, 2.0))
    if kind == "quadtree":
        return _case(None, kind, (rng.randint(1, 6), rng.randint(12, 36), rng.randint(16, 40)), logu(1e2, 1e5),
                     precision, rng.choice((0, 10)), wells=max(1, wells))
    uniform = rng.random() < 0.5
    shape = (logu(1, 20), logu(20, 200), logu(20, 200))
    times = 0 if kind in ("paths", "coupled") else rng.choice((0, rng.randint(1, 50)))
    n = {"paths": logu(1e2, 2e4), "batch": logu(4e3, 2.5e5), "host": logu(1e3, 2e5), "coupled": logu(1e2, 5e4),
         "periods": logu(1e2, 2e5), "track": logu(1e2, 1e6)}[kind]
    return _case(None, kind, shape, n, precision, times, var, wells, uniform,
                 rng.randint(8, 32) if kind == "batch" else 1)


# ---- inputs -----------------------------------------------------------------------


def _lognormal(shape, corr, var, gen):
    """K with exponential covariance, by circulant embedding on the GPU."""
    if var == 0.0:
        return torch.full(shape, 1e-4, dtype=torch.float64, device="cuda")
    pad = [s + int(math.ceil(4 * l)) for s, l in zip(shape, corr)]
    r2 = 0.0
    for a, (m, l) in enumerate(zip(pad, corr)):
        d = torch.arange(m, dtype=torch.float64, device="cuda")
        d = torch.minimum(d, m - d) / l
        r2 = r2 + (d * d).reshape([m if b == a else 1 for b in range(3)])
    eig = torch.fft.fftn(torch.exp(-torch.sqrt(r2))).real.clamp_(min=0.0)
    w = torch.randn(pad, dtype=torch.float64, device="cuda", generator=gen)
    y = torch.fft.ifftn(torch.sqrt(eig) * torch.fft.fftn(w)).real[:shape[0], :shape[1], :shape[2]]
    return torch.exp(LNK_MEAN + math.sqrt(var) * y)


def _solve(f, K, drop, q_src):
    """Face flows of a finite-volume head solve (conjugate gradients, diagonal
    preconditioner) with head `drop` + 10 m west and 10 m east."""
    dx, dy, dz = (torch.as_tensor(v, device="cuda") for v in (f.delr, f.delc, f.dz))
    rx, ry, rz = dx[None, None, :] / K / 2, dy[None, :, None] / K / 2, dz[:, None, None] / K / 2
    cx = (dy[None, :, None] * dz[:, None, None]) / (rx[:, :, 1:] + rx[:, :, :-1])
    cy = (dx[None, None, :] * dz[:, None, None]) / (ry[:, 1:] + ry[:, :-1])
    cz = (dx[None, None, :] * dy[None, :, None]) / (rz[1:] + rz[:-1])
    diag = torch.zeros_like(K)
    diag[:, :, 1:] += cx
    diag[:, :, :-1] += cx
    diag[:, 1:] += cy
    diag[:, :-1] += cy
    diag[1:] += cz
    diag[:-1] += cz
    free = torch.ones_like(K)
    free[:, :, 0] = free[:, :, -1] = 0.0
    inv = free / diag

    def flows(h):
        return cx * (h[:, :, :-1] - h[:, :, 1:]), cy * (h[:, :-1] - h[:, 1:]), cz * (h[:-1] - h[1:])

    def net(h):   # outflow of every free cell
        qx, qy, qz = flows(h)
        s = torch.zeros_like(h)
        s[:, :, :-1] += qx
        s[:, :, 1:] -= qx
        s[:, :-1] += qy
        s[:, 1:] -= qy
        s[:-1] += qz
        s[1:] -= qz
        return s * free

    x = torch.linspace(0.0, 1.0, K.shape[2], dtype=torch.float64, device="cuda")
    h = ((1.0 - x) * drop + 10.0).expand(K.shape).clone()
    r = (q_src - net(h)) * free
    z = r * inv
    p = z.clone()
    rz_ = (r * z).sum()
    first = rz_.clone()
    for it in range(12000):
        ap = net(p)
        alpha = rz_ / (p * ap).sum()
        h += alpha * p
        r -= alpha * ap
        torch.mul(r, inv, out=z)
        new = (r * z).sum()
        if it % 100 == 99 and float(new) <= 1e-22 * float(first):
            break
        p.mul_(new / rz_).add_(z)
        rz_ = new
    qx, qy, qz = flows(h)
    pad = torch.nn.functional.pad
    return pad(qx, (1, 1)), pad(qy, (0, 0, 1, 1)), pad(qz, (0, 0, 0, 0, 1, 1))


def _aquifer(case, seed, periods=1):
    """The flow fields of `periods` stress periods on one grid."""
    shape = (case["nlay"], case["nrow"], case["ncol"])
    gen = torch.Generator("cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    if case["var"] == 0.0:
        size, corr = (10.0, 10.0, 10.0), None
    else:
        size, corr = (5.0, 5.0, 1.0), (2.0, 10.0, 10.0) if case["nlay"] <= 20 else (8.0, 8.0, 8.0)
    if case["uniform"]:
        delr, delc, dz = (np.full(m, s) for m, s in zip(shape[::-1], size))
    else:
        delr, delc, dz = rng.uniform(1, 3, shape[2]), rng.uniform(1, 3, shape[1]), rng.uniform(0.5, 2, shape[0])
    K = _lognormal(shape, corr, case["var"], gen)
    por = torch.full(shape, POROSITY, dtype=torch.float64, device="cuda")
    if case["nlay"] > 20:
        por.uniform_(0.2, 0.35, generator=gen)
    ib = torch.ones(shape, dtype=torch.int8, device="cuda")
    ib[:, :, 0] = ib[:, :, -1] = -1
    q = torch.zeros_like(K)
    Lx = float(delr.sum())
    through = math.exp(LNK_MEAN) * float(delc.sum() * dz.sum())
    out = []
    for p in range(periods):
        for _ in range(case["wells"]):
            k, i, j = rng.integers(0, shape[0]), rng.integers(0, shape[1]), rng.integers(2, shape[2] - 2)
            ib[k, i, j] = 2
            q[k, i, j] = -float(rng.uniform(0.005, 0.02)) * through
        f = SimpleNamespace(nlay=shape[0], nrow=shape[1], ncol=shape[2], delr=delr, delc=delc, dz=dz,
                            origin=(0.0, 0.0, 0.0), porosity=por, ibound=ib.clone())
        f.qx, f.qy, f.qz = _solve(f, K, Lx * (1.0, 0.6, 1.3)[p % 3], q)
        out.append(f)
    torch.cuda.synchronize()
    return out


def _t_adv(case, f):
    """Mean advective crossing time at unit gradient."""
    return float(f.delr.sum()) * POROSITY / (1e-4 if case["var"] == 0.0 else math.exp(LNK_MEAN))


def _times(case, f):
    if not case["times"]:
        return None
    ta = _t_adv(case, f)
    return np.logspace(math.log10(ta / 100), math.log10(10 * ta), case["times"])


def _boxes(case, f, rng):
    """The release boxes (n, lo, hi, key) of a case's requests: a plane or a slab near the inflow side for one
    request, boxes anywhere for a batch, whose sizes are spread over their logarithm."""
    x = np.concatenate([[0.0], np.cumsum(f.delr)])
    Ly, Lz = float(f.delc.sum()), float(f.dz.sum())
    if case["kind"] != "batch":
        x1 = float(x[1])
        hi = float(x[min(6, f.ncol - 2)]) if case["var"] == 0.0 else x1
        return [(case["n"], (x1, 0.0, 0.0), (hi, Ly, Lz), int(rng.integers(1, 2 ** 62)))]
    share = np.exp(rng.uniform(0.0, math.log(200.0), case["reqs"]))
    sizes = np.maximum(1, (share / share.sum() * case["n"]).astype(int))
    sizes[-1] += case["n"] - int(sizes.sum())
    out, ext = [], (float(x[-2] - x[1]), Ly, Lz)
    for m in sizes:
        e = [float(rng.uniform(0.05, 0.5)) * v for v in ext]
        lo = [float(rng.uniform(0.0, v - w)) for v, w in zip(ext, e)]
        lo[0] += float(x[1])
        out.append((int(m), tuple(lo), tuple(a + b for a, b in zip(lo, e)), int(rng.integers(1, 2 ** 62))))
    return out


def _explicit(case, f, seed, gen):
    """n particles in active cells of the western fifth, as (cell, local fractions), on the GPU."""
    shape, n = (f.nlay, f.nrow, f.ncol), case["n"]
    j = torch.randint(1, max(2, f.ncol // 5), (n,), device="cuda", generator=gen)
    i = torch.randint(0, f.nrow, (n,), device="cuda", generator=gen)
    k = torch.randint(0, f.nlay, (n,), device="cuda", generator=gen)
    cell = ((k * shape[1] + i) * shape[2] + j).to(torch.int32)
    return cell, torch.rand((n, 3), dtype=torch.float64, device="cuda", generator=gen)


@functools.lru_cache(1)
def _context():
    return mp.Context(0)


class _Plan:
    """A loaded field (or several) and what goes with it; frees the fields with itself."""

    def __init__(self, case, seed):
        self.case, self.ctx = case, _context()
        rng = np.random.default_rng(seed + 1)
        gen = torch.Generator("cuda").manual_seed(seed + 1)
        kind, n, nt = case["kind"], case["n"], case["times"]
        self.opts = {"mode": mp.MODE_ENDPOINT | (mp.MODE_TIMESERIES if nt else 0),
                     "precision": mp.PREC_FP64 if case["precision"] == FP64 else mp.PREC_MIXED}
        self.cell = self.local = self.t0 = self.t_end = None
        self.flags, self.t_stop, self.boxes = 0, INF, None
        if kind == "quadtree":
            self.fields = [usg.quadtree_field(case["nlay"], case["nrow"], case["ncol"], seed, n_wells=case["wells"])]
            cell, local = usg.explicit_particles(self.fields[0], n, seed + 1)
            self.cell, self.local = torch.from_numpy(cell).cuda(), torch.from_numpy(local).cuda()
            ta = self.fields[0].extent[0] * 0.3 / 1e-4
            self.times = np.logspace(math.log10(ta / 100), math.log10(10 * ta), nt) if nt else None
            self.handles = [self.ctx.field(self.fields[0])]
        else:
            self.fields = _aquifer(case, seed, 3 if kind == "periods" else 1)
            f = self.fields[0]
            ta = _t_adv(case, f)
            self.times = _times(case, f)
            self.handles = [] if kind == "coupled" else [self.ctx.field(g, device_arrays=True) for g in self.fields]
            if kind in ("paths", "coupled", "periods", "host"):
                self.cell, self.local = _explicit(case, f, seed, gen)
            if kind == "paths":      # ten stages over a fifth of the crossing time
                self.t0 = torch.arange(n, device="cuda").remainder(10).double() * (ta / 50)
                self.opts["mode"] |= mp.MODE_PATHLINE
                self.opts["path_capacity"] = n * (3 * case["ncol"] + 50)   # about twice what the paths need
            elif kind == "periods":
                self.t_end = [0.2 * ta, 0.6 * ta]
                self.flags = mp.TRACK_PASS_WEAK_SINKS
            elif kind == "coupled":
                self.t_stop = 0.25 * ta
            elif kind == "host":
                self.cell, self.local = self.cell.cpu().numpy(), self.local.cpu().numpy()
            if kind in ("track", "batch"):
                self.boxes = _boxes(case, f, rng)
        self.opts.update(times=self.times, t_stop=self.t_stop, flags=self.flags)
        if kind == "host":   # a host program keeps its result arrays from call to call
            self.out = {k: np.empty(n, d) for k, d in mp.ENDPOINT_DTYPES.items()}
            self.ts = np.empty((nt, n), mp.TS_RECORD) if nt else None
        else:
            kinds = {np.int32: torch.int32, np.float64: torch.float64, np.uint8: torch.uint8,
                     np.uint32: torch.int32, np.uint64: torch.int64}
            self.out = {k: torch.empty(n, dtype=kinds[d], device="cuda") for k, d in mp.ENDPOINT_DTYPES.items()}
            self.ts = torch.empty((nt * n, 4), dtype=torch.float64, device="cuda") if nt else None
            if kind == "paths":
                self.points = torch.empty((self.opts["path_capacity"], 6), dtype=torch.float64, device="cuda")

    def __del__(self):
        try:
            torch.cuda.synchronize()
            for h in self.handles:
                mp.mp_field_free(h)
        except Exception:   # interpreter shutdown
            pass


def prepare(case, seed):
    return _Plan(case, seed)


# ---- one pass ---------------------------------------------------------------------


def _result(out, ts, more=None):
    """Endpoint arrays by name, the timeseries records as positions, cells and statuses."""
    res = dict(out)
    if ts is not None:
        whole = ts.view(torch.int32)
        res["ts_pos"], res["ts_cell"], res["ts_status"] = ts[:, :3], whole[:, 6], whole[:, 7]
    return {**res, **(more or {})}


def run(s):
    kind, ctx = s.case["kind"], s.ctx
    if kind == "host":
        out, ts, _ = mp.mp_track_host(ctx.h, s.handles[0], s.cell, s.local, mp.make_opts(**s.opts), out=s.out,
                                      ts_out=s.ts)
        return _result({k: (v.view("i4") if v.dtype == np.uint32 else v.view("i8") if v.dtype == np.uint64 else v)
                        for k, v in out.items()},
                       None if ts is None else torch.from_numpy(ts.view("f8").reshape(-1, 4)))
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "batch":
        opts = mp.make_opts(**s.opts)
        groups = [ctx.release_box(s.handles[0], m, lo, hi, key, stream=stream) for m, lo, hi, key in s.boxes]
        ids = mp.mp_track_batch(ctx.h, groups, [opts] * len(groups), stream)
        at = 0
        for g, r, (m, _, _, _) in zip(groups, ids, s.boxes):
            mp.mp_get_endpoints(ctx.h, r, m, out={k: v[at:] for k, v in s.out.items()}, device=True, stream=stream)
            if s.ts is not None:   # each request's records follow the ones before
                mp.mp_get_timeseries(ctx.h, r, m, s.case["times"], out=s.ts[at * s.case["times"]:], device=True,
                                     stream=stream)
            at += m
            mp.mp_req_free(ctx.h, r)
            mp.mp_group_free(g)
        return _result(s.out, s.ts)
    if kind == "coupled":
        fh = ctx.field(s.fields[0], device_arrays=True)
    else:
        fh = s.handles[0]
    if s.boxes is not None:
        n, lo, hi, key = s.boxes[0]
        g = ctx.release_box(fh, n, lo, hi, key, stream=stream)
    else:
        g = ctx.release_explicit(fh, s.cell, s.local, s.t0, stream=stream, device_arrays=True)
    if kind == "periods":
        req = ctx.track_periods(g, s.handles, s.t_end, stream=stream, **s.opts)
    else:
        req = ctx.track(g, stream=stream, **s.opts)
    mp.mp_get_endpoints(ctx.h, req.id, req.n, out=s.out, device=True, stream=stream)
    if s.ts is not None:
        mp.mp_get_timeseries(ctx.h, req.id, req.n, req.n_times, out=s.ts, device=True, stream=stream)
    more = {}
    if kind == "paths":
        m = min(req.stats()["path_points"], s.points.shape[0])
        mp.mp_get_pathlines(ctx.h, req.id, m, out=s.points, device=True, stream=stream)
        whole = s.points[:m].view(torch.int32)
        order = torch.argsort(whole[:, 8].long() << 32 | whole[:, 10].long())
        pts = torch.zeros_like(s.points)   # the unused rows stay zero
        torch.index_select(s.points, 0, order, out=pts[:m])
        whole = pts.view(torch.int32)
        more = {"path_pos": pts[:, :4], "path_id": whole[:, 8:11], "path_status": whole[:, 11]}
    if kind == "coupled":
        more = mp.mp_field_balance(fh)
    req.free()
    mp.mp_group_free(g)
    if kind == "coupled":
        mp.mp_field_free(fh)
    return _result(s.out, s.ts, more)


def work(case):
    """Field and results once; about 200 floating operations a cell-step, 1.4 steps a column crossed."""
    cells, n = case["nlay"] * case["nrow"] * case["ncol"], case["n"]
    part = {"coupled": 0.2, "batch": 0.6, "periods": 0.85, "paths": 0.85, "host": 0.85}.get(case["kind"], 1.0)
    steps = n * (1.0 + 1.4 * part * case["ncol"])
    field = cells * {"quadtree": 260, "coupled": 34, "periods": 99}.get(case["kind"], 33)
    points = 96 * steps if case["kind"] == "paths" else 0
    return {"bytes": field + n * (74 + 32 * case["times"]) + points, "flops": 200.0 * steps}


# ---- the same in 64 bits, from the statement of the method ---------------------------


def _philox(n, seed):
    """Three uniforms per particle: Philox4x32-10 on counters (q, 0 or 1) under the key `seed`."""
    def block(last):
        c = [np.arange(n, dtype=np.uint64), np.zeros(n, np.uint64), np.full(n, last, np.uint64), np.zeros(n, np.uint64)]
        k, low, half = [seed & 0xFFFFFFFF, seed >> 32], np.uint64(0xFFFFFFFF), np.uint64(32)
        for _ in range(10):
            a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
            c = [b >> half ^ c[1] ^ np.uint64(k[0]), b & low, a >> half ^ c[3] ^ np.uint64(k[1]), a & low]
            k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
        return c

    def unit(a, b):
        return ((a << np.uint64(32) | b) >> np.uint64(11)).astype(np.float64) / 2.0 ** 53

    r, s = block(0), block(1)
    return np.stack([unit(r[0], r[1]), unit(r[2], r[3]), unit(s[0], s[1])], 1)


def _pollock(v1, v2, D, p):
    """Per axis: velocity, gradient, reachable face (+1, -1, 0) and the time to it."""
    A = (v2 - v1) / D
    v = v1 + A * p
    face = torch.where((v > 0) & (v2 > 0), 1, torch.where((v < 0) & (v1 < 0), -1, 0))
    t = torch.where(face > 0, D - p, -p) / torch.where(face == 0, 1.0, v)
    z = A * t
    t = torch.where(z == 0, t, t * torch.log1p(torch.where(z == 0, 0.5, z)) / torch.where(z == 0, 1.0, z))
    return v, A, face, torch.where(face == 0, INF, t)


def _moved(v, A, D, p, dt):
    w = A * dt
    f = torch.where(w == 0, 1.0, torch.expm1(torch.where(w == 0, 0.5, w)) / torch.where(w == 0, 1.0, w))
    return torch.where((v == 0) | (dt == 0), p, torch.minimum((p + v * dt * f).clamp(min=0.0), D))


def _follow(fields, ends, ijk, p, t0, times, t_stop, pass_sinks, order):
    """Pollock's displacement, cell by cell, for all particles at once.  `order` maps a particle's record of output
    time k to a row of the records."""
    dev, f0 = "cuda", fields[0]
    dims = torch.tensor([f0.ncol, f0.nrow, f0.nlay], device=dev)
    size = [torch.as_tensor(v, device=dev) for v in (f0.delr, f0.delc, f0.dz)]
    edge = [torch.as_tensor(np.concatenate([[0.0], np.cumsum(v)]), device=dev) for v in (f0.delr, f0.delc, f0.dz)]
    n, nt = p.shape[0], 0 if times is None else len(times)
    tk = torch.as_tensor(np.append(times if nt else [], INF), device=dev)
    t, ijk, p = t0.clone(), ijk.clone(), p.clone()
    alive = torch.ones(n, dtype=torch.bool, device=dev)
    kn = torch.zeros(n, dtype=torch.long, device=dev)
    rec = torch.zeros((nt * n, 3), dtype=torch.float64, device=dev)

    def place(i, q):
        return torch.stack([edge[a][ijk[i, a]] + q[:, a] for a in range(3)], 1)

    def write(i, q, until):   # the records of particles i at q up to the times `until`
        while True:
            due = tk[kn[i]] <= until
            if not due.any():
                return
            j = i[due]
            rec[order(j, kn[j])] = place(j, q[due])
            kn[j] += 1

    everyone = torch.arange(n, device=dev)
    ib0 = f0.ibound[ijk[:, 2], ijk[:, 1], ijk[:, 0]]
    alive &= ib0 == 1
    if nt:
        write(everyone, p, t)
    for number, f in enumerate(fields):
        stop = t_stop if number == len(fields) - 1 else min(t_stop, ends[number])
        area = (size[1][None, :, None] * size[2][:, None, None], size[0][None, None, :] * size[2][:, None, None],
                size[0][None, None, :] * size[1][None, :, None])
        lo = [q / (f.porosity * a) for q, a in zip((f.qx[:, :, :-1], f.qy[:, :-1], f.qz[:-1]), area)]
        hi = [q / (f.porosity * a) for q, a in zip((f.qx[:, :, 1:], f.qy[:, 1:], f.qz[1:]), area)]
        here = f.ibound[ijk[:, 2], ijk[:, 1], ijk[:, 0]]
        alive &= (here == 1) | ((here == 2) & pass_sinks)
        go = alive & (t < stop)
        while True:
            i = go.nonzero()[:, 0]
            if not i.numel():
                break
            c = ijk[i]
            at = (c[:, 2], c[:, 1], c[:, 0])
            D = [size[a][c[:, a]] for a in range(3)]
            parts = [_pollock(lo[a][at], hi[a][at], D[a], p[i, a]) for a in range(3)]
            te = torch.stack([x[3] for x in parts], 1)
            te = torch.where(torch.isnan(te), INF, te)
            dt, ax = te.min(1)
            ax = torch.where(te[:, 0] == dt, 0, torch.where(te[:, 1] == dt, 1, 2))   # the lowest axis on ties
            stuck = torch.isinf(dt)
            caught = stuck & (f.ibound[at] == 2)
            end = t[i] + dt
            ends_here = ~caught & (stuck | (end >= stop)) if stop < INF else torch.zeros_like(stuck)
            lost = caught | (stuck & ~ends_here)
            until = torch.where(ends_here, stop, end)
            until = torch.where(caught, -INF, until)
            if nt:
                while True:
                    due = tk[kn[i]] <= until
                    if not due.any():
                        break
                    j, tau = i[due], tk[kn[i[due]]] - t[i[due]]
                    q = torch.stack([_moved(x[0][due], x[1][due], D[a][due], p[j, a], tau)
                                     for a, x in enumerate(parts)], 1)
                    rec[order(j, kn[j])] = place(j, q)
                    kn[j] += 1
            step = torch.where(ends_here, stop - t[i], torch.where(lost, 0.0, dt))
            q = torch.stack([_moved(x[0], x[1], D[a], p[i, a], step) for a, x in enumerate(parts)], 1)
            face = torch.stack([x[2] for x in parts], 1)[torch.arange(i.numel(), device=dev), ax]
            cross = ~ends_here & ~lost
            rows = cross.nonzero()[:, 0]
            q[rows, ax[rows]] = torch.where(face[rows] > 0, torch.stack(D, 1)[rows, ax[rows]], 0.0)
            p[i] = q
            t[i] = torch.where(ends_here, stop, torch.where(lost, t[i], end))
            go[i[ends_here]] = False
            alive[i[lost]] = False
            # into the neighbour, unless it ends the path
            to = c[rows].clone()
            to[torch.arange(rows.numel(), device=dev), ax[rows]] += face[rows]
            inside = ((to >= 0) & (to < dims)).all(1)
            safe = torch.where(inside[:, None], to, 0)
            kind = f.ibound[safe[:, 2], safe[:, 1], safe[:, 0]]
            enter = inside & ((kind == 1) | ((kind == 2) & pass_sinks))
            alive[i[rows[~enter]]] = False
            w, a = i[rows[enter]], ax[rows[enter]]
            ijk[w] = to[enter]
            far = torch.stack([size[b][to[enter][:, b]] for b in range(3)], 1)
            p[w, a] = torch.where(face[rows[enter]] < 0, far[torch.arange(w.numel(), device=dev), a], 0.0)
            go &= alive
    x = place(everyone, p)
    for k in range(nt):
        j = everyone[kn <= k]
        rec[order(j, torch.full_like(j, k))] = x[j]
    return x, p, t, rec


def exact(case, seed):
    kind = case["kind"]
    if kind == "quadtree":
        return None   # no plain form of the refined grid's hand-over here
    s = prepare(case, seed)
    f, n, nt = s.fields[0], case["n"], case["times"]
    if s.boxes is not None:
        pts = torch.from_numpy(np.concatenate(
            [np.asarray(lo) + _philox(m, key) * (np.asarray(hi) - np.asarray(lo)) for m, lo, hi, key in s.boxes])).cuda()
        edges = [torch.as_tensor(np.concatenate([[0.0], np.cumsum(v)]), device="cuda") for v in (f.delr, f.delc, f.dz)]
        ijk = torch.stack([(torch.searchsorted(e, pts[:, a].contiguous(), right=True) - 1).clamp(0, e.numel() - 2)
                           for a, e in enumerate(edges)], 1)
        p = pts - torch.stack([e[ijk[:, a]] for a, e in enumerate(edges)], 1)
        t0 = torch.zeros(n, dtype=torch.float64, device="cuda")
    else:
        cell = torch.as_tensor(s.cell, device="cuda").long()
        row = cell // f.ncol
        ijk = torch.stack([cell % f.ncol, row % f.nrow, row // f.nrow], 1)
        p = torch.as_tensor(s.local, device="cuda") * torch.stack(
            [torch.as_tensor(v, device="cuda")[ijk[:, a]] for a, v in enumerate((f.delr, f.delc, f.dz))], 1)
        t0 = torch.zeros(n, dtype=torch.float64, device="cuda") if s.t0 is None else s.t0
    if s.boxes is not None and len(s.boxes) > 1:   # each request's records follow the ones before
        m = torch.tensor([b[0] for b in s.boxes], device="cuda")
        own, start = torch.repeat_interleave(m, m), torch.repeat_interleave(m.cumsum(0) - m, m)
        order = lambda j, k: start[j] * nt + k * own[j] + (j - start[j])  # noqa: E731
    else:
        order = lambda j, k: k * n + j  # noqa: E731
    x, p, t, rec = _follow(s.fields, s.t_end, ijk, p, t0, s.times, s.t_stop, bool(s.flags), order)
    out = {k: None for k in mp.ENDPOINT_DTYPES}
    out.update(x=x[:, 0], y=x[:, 1], z=x[:, 2], t=t)
    if case["precision"] == FP64:   # (a mixed-precision path may end in the next cell: another offset for the same place)
        out.update(px=p[:, 0], py=p[:, 1], pz=p[:, 2])
    if nt:
        out["ts_pos"] = rec
    return out
