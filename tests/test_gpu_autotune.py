"""What mp_autotune keeps: nothing from a sample that every candidate tracks
with the same few-particle kernel, never a launch slower than the one chosen
without it, and nothing beyond the field it was measured on."""
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


@pytest.mark.parametrize("precision,few", [(mp.PREC_FP64, 18240), (mp.PREC_MIXED, 30400)])
@pytest.mark.parametrize("sample", [False, True])
def test_few_particles_store_nothing(ctx, precision, few, sample):
    w = I.workload("cfg1")
    fh = ctx.field(w.field)
    n = few if not sample else 40000
    gh = ctx.release_box(fh, n, w.release.lo, w.release.hi, 5)
    many = ctx.release_box(fh, 40000, w.release.lo, w.release.hi, 6)
    mp.mp_set_tuning(ctx.h, fh, precision, False, SLOW)
    assert _ms(ctx, many, precision, mp.SCHED_AUTO) > 20.0
    t = mp.mp_autotune(ctx.h, gh, mp.make_opts(precision=precision), sample=1000 if sample else 0)
    assert t["tried"] == 1 and t["ms"] > 0.0 and 32 <= t["block"] <= 256
    assert _ms(ctx, many, precision, mp.SCHED_AUTO) > 20.0
    mp.mp_set_tuning(ctx.h, fh, precision, False, t)      # the result is one that can be installed
    assert _ms(ctx, many, precision, mp.SCHED_AUTO) < 20.0


@pytest.mark.parametrize("precision", [mp.PREC_FP64, mp.PREC_MIXED])
def test_tuned_is_not_slower_than_untuned(ctx, precision):
    f = I.random_box_field(20, 100, 100, seed=5, lnk_var=1.0, n_wells=4)
    fh = ctx.field(f)
    cells, frac = I.explicit_particles(f, 60000, seed=3, cols=(1, 5))
    gh = ctx.release_explicit(fh, cells, frac)
    untuned = _ms(ctx, gh, precision, mp.SCHED_DYNAMIC, 9)
    t = mp.mp_autotune(ctx.h, gh, mp.make_opts(precision=precision))
    assert t["tried"] == 13
    tuned = _ms(ctx, gh, precision, mp.SCHED_AUTO, 9)
    # (medians of nine launches lie within 1 % of each other)
    assert tuned <= 1.02 * untuned, (tuned, untuned, t)


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
