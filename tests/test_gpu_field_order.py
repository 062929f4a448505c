"""mp_field_load with device arrays reads what the work enqueued before the
call writes: on the default stream, and through the Python binding on torch's
current stream, with no host synchronisation in between."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu


def _field(torch, q):
    shape = (4, 60, 60)
    f = SimpleNamespace(nlay=4, nrow=60, ncol=60, delr=np.ones(60), delc=np.ones(60), dz=np.ones(4),
                        origin=(0.0, 0.0, 0.0), porosity=torch.full(shape, 0.3, dtype=torch.float64, device="cuda"),
                        ibound=torch.ones(shape, dtype=torch.int8, device="cuda"))
    f.qx, f.qy, f.qz = (torch.full(s, q, dtype=torch.float64, device="cuda") for s in ((4, 60, 61), (4, 61, 60), (5, 60, 60)))
    f.qx[0, 0, 0] = 10.0 * q
    f.ibound[0, 0, 0] = 2                                 # extracts 9 q
    return f


@pytest.mark.parametrize("side", [False, True])
def test_load_after_the_producer(side):
    import torch
    # (whether two streams share a hardware queue, and so run in order by
    # chance, differs from context to context)
    for _ in range(6):
        with mp.Context(0) as ctx:
            mp.mp_field_free(ctx.field(_field(torch, 1.0), device_arrays=True))
            f = _field(torch, 1.0)
            torch.cuda.synchronize()
            with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.default_stream()):
                torch.cuda._sleep(40_000_000)             # some 20 ms, then the new flows
                for q in (f.qx, f.qy, f.qz):
                    q.mul_(2.0)
                fh = ctx.field(f, device_arrays=True)
            assert mp.mp_field_balance(fh)["sink_extraction"] == 18.0
            mp.mp_field_free(fh)
