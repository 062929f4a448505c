"""What mp_autotune and mp_set_tuning keep: nothing beyond the field that it
belongs to."""
import numpy as np
import pytest

from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu

# an installed launch that shows: warps that fetch again only after two million steps take over 20 ms
SLOW = {"schedule": mp.SCHED_DYNAMIC, "block": 32, "steps_per_fetch": 2_000_000}


@pytest.fixture()
def ctx():
    import torch  # noqa: F401
    c = mp.Context(0)
    yield c
    c.close()


def _ms(ctx, gh, precision, schedule, reps=1):
    out = []
    for _ in range(reps):
        r = ctx.track(gh, precision=precision, schedule=schedule)
        out.append(r.stats()["kernel_ms"])
        r.free()
    return float(np.median(out))


def test_tuning_goes_with_its_field(ctx):
    w = I.workload("cfg1")
    fh = ctx.field(w.field)
    mp.mp_set_tuning(ctx.h, fh, mp.PREC_FP64, False, SLOW)
    gh = ctx.release_box(fh, 40000, w.release.lo, w.release.hi, 5)
    assert _ms(ctx, gh, mp.PREC_FP64, mp.SCHED_AUTO) > 20.0
    mp.mp_group_free(gh)
    old = fh.value
    mp.mp_field_free(fh)
    kept = []
    for _ in range(200):                                  # until a new field has the old one's address
        kept.append(ctx.field(w.field))
        if kept[-1].value == old:
            break
    else:
        pytest.skip("the address was not used again")
    gh = ctx.release_box(kept[-1], 40000, w.release.lo, w.release.hi, 5)
    assert _ms(ctx, gh, mp.PREC_FP64, mp.SCHED_AUTO) < 20.0
