"""The exit axis where its choice is delicate, FP64: a leading axis whose exact
exit time is not finite (the face velocity behind it is tiny, so 1 + z rounds
to zero), with the two other axes' times close together around the bound up to
which an estimate counts as a candidate.  The axis with the smallest exact
time wins, in launches of few particles and of many."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = mp.Context(0)
    yield c
    c.close()


def _endpoints(ctx, fh, cells, frac, **kw):
    g = ctx.release_explicit(fh, cells, frac)
    req = ctx.track(g, **kw)
    ep = req.endpoints()
    req.free()
    mp.mp_group_free(g)
    return ep


def test_leading_time_not_finite(ctx):
    n, rep, blocks = 16000, 2, 64                        # 16,000 particles: three lanes each; 32,000: one
    rng = np.random.default_rng(11)
    vx2, vy, vz2 = 2.0 ** -60, 0.012010, 0.01205
    nc, mid = 3 * blocks, 3 * np.arange(blocks) + 1       # one such cell in every third column
    T0 = -np.log(vx2) * (1.0 + 2.0 ** -10)
    gz = np.exp(rng.uniform(np.log(0.0079), np.log(0.3), blocks)) / T0
    q = [np.full(s, 1e-3) for s in ((3, 3, nc + 1), (3, 4, nc), (4, 3, nc))]
    q[0][1, 1, mid], q[0][1, 1, mid + 1] = 1.0, vx2       # x: velocity 1 -> 2^-60, exact time infinite
    q[1][1, 1:3, mid] = vy                                # y: constant velocity
    q[2][1, 1, mid], q[2][2, 1, mid] = vz2 - gz, vz2      # z: a gradient, z = A t1 from just above 2^-7 on
    f = SimpleNamespace(nlay=3, nrow=3, ncol=nc, delr=np.ones(nc), delc=np.ones(3), dz=np.ones(3),
                        origin=(0.0, 0.0, 0.0), qx=q[0], qy=q[1], qz=q[2], porosity=np.ones((3, 3, nc)),
                        ibound=np.ones((3, 3, nc), np.int8))
    at = rng.integers(0, blocks, n)
    # both times near the bound, at distances over three decades
    T = T0 * (1.0 + rng.choice([-1.0, 1.0], (2, n)) * np.exp(rng.uniform(np.log(3e-8), np.log(3e-5), (2, n))))
    frac = np.stack([np.zeros(n), 1.0 - vy * T[0], 1.0 + vz2 * np.expm1(-gz[at] * T[1]) / gz[at]], 1)
    ty = (1.0 - frac[:, 1]) / vy
    A = vz2 - (vz2 - gz[at])
    tz = -np.log1p(-A * (1.0 - frac[:, 2]) / vz2) / A
    clear = np.abs(ty - tz) > 1e-11 * ty
    cells = ((1 * 3 + 1) * nc + mid[at]).astype(np.int32)
    want = np.where(ty < tz, cells + nc, cells + 3 * nc)   # the cell entered
    fh = ctx.field(f)
    few = _endpoints(ctx, fh, cells, frac, max_steps=1)
    many = _endpoints(ctx, fh, np.tile(cells, rep), np.tile(frac, (rep, 1)), max_steps=1)
    assert clear.sum() > 0.99 * n and 0.3 * n < (ty < tz).sum() < 0.7 * n
    for k, v in few.items():
        assert np.array_equal(many[k].reshape(rep, n)[rep - 1].view(np.uint8), v.view(np.uint8)), k
    assert np.array_equal(few["cell"][clear], want[clear])
    mp.mp_field_free(fh)
