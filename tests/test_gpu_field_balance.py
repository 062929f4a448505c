"""The volume balance reduced on the device equals the sums over the cells
in order, exactly, for grids at the edges of its tiles and runs, with no
sinks, single ones, whole runs of them, and inactive cells."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2302_13590_gb300 import mp
from tests.test_gpu_parity import _balance_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = mp.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("ncol,sinks", [(1, "none"), (255, "some"), (256, "all but one"), (257, "last"), (1000, "some"),
                                        (262144, "some"), (262145, "runs"), (524545, "some")])
def test_balance_equals_sums_in_cell_order(ctx, ncol, sinks, device):
    import torch
    rng = np.random.default_rng(ncol)
    q = [rng.standard_normal(s) * 1e-4 for s in ((1, 1, ncol + 1), (1, 2, ncol), (2, 1, ncol))]
    ib = rng.choice(np.array([-1, 0, 1, 1, 1], np.int8), ncol)
    if sinks == "some":
        ib[rng.random(ncol) < 0.01] = 2
    elif sinks == "all but one":
        ib[:] = 2
    elif sinks == "last":
        ib[-1] = 2
    elif sinks == "runs":
        ib[rng.random(ncol) < 0.5] = 2
        ib[1024:4096] = 2
    ib[ncol // 2] = 1
    f = SimpleNamespace(nlay=1, nrow=1, ncol=ncol, delr=np.ones(ncol), delc=np.ones(1), dz=np.ones(1),
                        origin=(0.0, 0.0, 0.0), qx=q[0], qy=q[1], qz=q[2], porosity=np.full(ncol, 0.3), ibound=ib)
    ref = _balance_np(np.stack([q[0][0, 0, :-1], q[0][0, 0, 1:], q[1][0, 0], q[1][0, 1], q[2][0, 0], q[2][1, 0]], -1), ib)
    if device:
        for k in ("qx", "qy", "qz", "porosity", "ibound"):
            setattr(f, k, torch.from_numpy(getattr(f, k)).cuda())
        torch.cuda.synchronize()
    for _ in range(2):   # the second load reuses the first one's memory
        fh = ctx.field(f, device_arrays=device)
        assert mp.mp_field_balance(fh) == ref
        mp.mp_field_free(fh)
