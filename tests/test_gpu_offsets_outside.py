"""Particles handed in with offsets outside their cell (rounded by the caller,
or further out): the exit time to the face behind is negative and the smallest
one wins, as the oracle has it, in launches of few particles and of many, bit
for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu

TORCH = {np.int32: "int32", np.float64: "float64", np.uint8: "uint8", np.uint32: "int32", np.uint64: "int64"}


@pytest.mark.parametrize("n", [10, 257])
@pytest.mark.parametrize("axes", [1, 3])
@pytest.mark.parametrize("past", [1e-13, 1e-6, 0.2])
def test_offsets_outside_the_cell(n, axes, past):
    import torch
    f = I.random_box_field(5, 19, 23, seed=61, lnk_var=2.5, n_wells=6, n_inactive=9, well_scale=4.0)
    cells, frac = I.explicit_particles(f, n, seed=n + 7)
    rng = np.random.default_rng(n)
    state = O.release_explicit(f, cells, frac)
    c = state["cell"]
    size = {"px": f.delr[c % f.ncol], "py": f.delc[c // f.ncol % f.nrow], "pz": f.dz[c // (f.ncol * f.nrow)]}
    first = rng.integers(0, 3, n)
    for a, k in enumerate(("px", "py", "pz")):
        move = (first == a) | (axes == 3)
        out = past * rng.uniform(0.5, 1.0, n)
        state[k] = np.where(move, size[k] * np.where(rng.random(n) < 0.5, -out, 1.0 + out), state[k])
    ref = O.track(f, state, arith="mirror")
    rep = 18240 // n + 1                                  # beyond what takes three lanes a particle
    with mp.Context(0) as ctx:
        fh = ctx.field(f)
        for copies in (1, rep):
            dev = {k: torch.from_numpy(np.tile(state[k], copies)).cuda() for k in ("cell", "px", "py", "pz", "t", "status")}
            out = {k: torch.empty(n * copies, dtype=getattr(torch, TORCH[d]), device="cuda")
                   for k, d in mp.ENDPOINT_DTYPES.items()}
            mp.mp_track_noalloc(fh, dev, out, opts=mp.make_opts())
            for k, d in mp.ENDPOINT_DTYPES.items():
                got = out[k].cpu().numpy().view(d).reshape(copies, n)
                want = ref[{"x": "gx", "y": "gy", "z": "gz"}.get(k, k)]
                assert np.array_equal(got[0], want, equal_nan=d is np.float64), (k, copies)
                assert np.array_equal(got[copies - 1], got[0], equal_nan=d is np.float64), (k, copies)
