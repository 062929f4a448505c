"""mp_field_free next to other streams: it does not disturb a capture that is
under way, and work already enqueued (a request whose id is gone, a release, a
launch without allocation) still reads the field that was freed behind it."""
import threading

import numpy as np
import pytest

from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp
from tests.test_zz_no_alloc import _device_out, _device_state

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    import torch  # noqa: F401
    c = mp.Context(0)
    yield c
    c.close()


def _flow(seed, **kw):
    return I.random_box_field(5, 40, 50, seed=seed, lnk_var=1.5, n_wells=4, **kw)


@pytest.mark.parametrize("mode,thread", [("relaxed", False), ("relaxed", True), ("thread_local", True)])
def test_free_while_a_stream_is_captured(ctx, mode, thread):
    import torch
    fh = ctx.field(_flow(1))
    x = torch.zeros(64, device="cuda")
    torch.cuda.synchronize()
    err = []

    def free():
        try:
            mp.mp_field_free(fh)
        except mp.MPError as e:
            err.append(e)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(torch.cuda.Stream()):
        g.capture_begin(capture_error_mode=mode)
        try:
            x.add_(1.0)
            if thread:
                t = threading.Thread(target=free)
                t.start()
                t.join()
            else:
                free()
            x.add_(1.0)
        finally:
            g.capture_end()
    g.replay()
    torch.cuda.synchronize()
    assert not err and float(x[0]) == 2.0


@pytest.mark.parametrize("what", ["request", "release", "noalloc"])
def test_memory_is_handed_on_after_the_work_behind_it(ctx, what):
    import torch
    a, b = _flow(2, n_inactive=300), _flow(3)
    n = 2000
    cells, frac = I.explicit_particles(a, n, seed=4, active_only=False)
    dcell, dfrac = torch.from_numpy(cells).cuda(), torch.from_numpy(frac.reshape(n, 3)).cuda()
    torch.cuda.synchronize()
    outs = []
    for late in (False, True):
        fh = ctx.field(a)
        stream = torch.cuda.Stream()
        out = _device_out(torch, n)
        if what == "noalloc":
            g = ctx.release_explicit(fh, cells, frac)
            r = ctx.track(g, t_stop=0.0)
            state = _device_state(torch, r.endpoints())
            r.free()
            mp.mp_group_free(g)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            if late:
                torch.cuda._sleep(60_000_000)             # some 30 ms
        h = stream.cuda_stream
        if what == "noalloc":
            mp.mp_track_noalloc(fh, state, out, opts=mp.make_opts(), stream=stream, want_stats=False)
        else:
            g = ctx.release_explicit(fh, dcell, dfrac, stream=h, device_arrays=True)
            if what == "request":
                r = ctx.track(g, stream=h)
                mp.mp_get_endpoints(ctx.h, r.id, n, out=out, device=True, stream=h)
                r.free()
                mp.mp_group_free(g)
        if not late:
            stream.synchronize()
        mp.mp_field_free(fh)
        fb = ctx.field(b)                                 # may take over the memory
        if what == "release":
            outs.append(None)
        stream.synchronize()
        if what == "release":                             # the statuses came from the first field's cell classes
            mp.mp_group_set_field(g, fb)
            r = ctx.track(g, t_stop=0.0)
            outs[-1] = r.endpoints()["status"]
            r.free()
            mp.mp_group_free(g)
        else:
            outs.append({k: v.cpu().numpy() for k, v in out.items()})
        mp.mp_field_free(fb)
    if what == "release":
        assert np.array_equal(outs[0], outs[1]) and (outs[0] == mp.ST_INVALID_RELEASE).any()
    else:
        for k in outs[0]:
            assert np.array_equal(outs[0][k].view(np.uint8), outs[1][k].view(np.uint8)), k
