"""Endpoint arrays read into device memory (one launch for all of them)
equal the host read at every size and start of a caller's slice, and leave
the memory around it alone; a batch whose requests have output times of
their own gives each request its own records."""
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


@pytest.mark.parametrize("n,off", [(1, 0), (1, 3), (15, 1), (16, 0), (17, 2), (1000, 5), (4099, 1), (70001, 7)])
def test_device_endpoints_equal_host_read(ctx, n, off):
    import torch
    f = I.cfg1_field()
    fh = ctx.field(f)
    cells, frac = I.explicit_particles(f, n, seed=n, cols=(1, 40))
    gh = ctx.release_explicit(fh, cells, frac)
    req = ctx.track(gh)
    want = req.endpoints()
    # `off` bytes (single-byte arrays) or elements into buffers of 0xa5, a guard behind
    bufs, out = {}, {}
    for k, dt in mp.ENDPOINT_DTYPES.items():
        size = np.dtype(dt).itemsize
        bufs[k] = torch.full(((n + off + 16) * size,), 0xa5, dtype=torch.uint8, device="cuda")
        out[k] = bufs[k][off * size:]
    out["t"] = bufs["t"][1:]   # not even a double's alignment
    mp.mp_get_endpoints(ctx.h, req.id, n, out=out, device=True)
    torch.cuda.synchronize()
    for k, dt in mp.ENDPOINT_DTYPES.items():
        size = np.dtype(dt).itemsize
        b = bufs[k].cpu().numpy()
        at = 1 if k == "t" else off * size
        assert np.array_equal(b[at:at + n * size], want[k].view(np.uint8)), k
        assert (b[:at] == 0xa5).all() and (b[at + n * size:] == 0xa5).all(), k
    req.free()
    mp.mp_group_free(gh)
    mp.mp_field_free(fh)


@pytest.mark.parametrize("precision", [mp.PREC_FP64, mp.PREC_MIXED])
def test_batch_with_times_of_each_request(ctx, precision):
    w = I.workload("cfg1")
    fh = ctx.field(w.field)
    shared = w.times[::7]
    times = [w.times[:1], shared, shared, None, w.times, w.times[::3], None, shared]
    groups = [ctx.release_box(fh, 50 + 31 * i, w.release.lo, w.release.hi, 9 + i) for i in range(len(times))]
    opts = [mp.make_opts(mode=mp.MODE_ENDPOINT | (mp.MODE_TIMESERIES if t is not None else 0), precision=precision,
                         times=t) for t in times]
    ids = mp.mp_track_batch(ctx.h, groups, opts)
    for i, (g, r, t) in enumerate(zip(groups, ids, times)):
        if t is not None:
            got = mp.mp_get_timeseries(ctx.h, r, 50 + 31 * i, len(t))
            alone = ctx.track(g, mode=mp.MODE_ENDPOINT | mp.MODE_TIMESERIES, precision=precision, times=t)
            assert np.array_equal(got.view(np.uint8), alone.timeseries().view(np.uint8)), i
            alone.free()
        mp.mp_req_free(ctx.h, r)
    for g in groups:
        mp.mp_group_free(g)
    mp.mp_field_free(fh)
