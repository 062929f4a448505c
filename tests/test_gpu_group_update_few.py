"""Launches of few particles that write the group's state back (whose three
lanes a particle all load it): particles that end at their start keep their
state and status, the others go on from where they stopped, as the oracle has
them."""
import numpy as np
import pytest

import oracle as O
from paper_2302_13590_gb300 import inputs as I
from paper_2302_13590_gb300 import mp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 10, 31, 4000])
def test_state_written_back_at_the_start(n):
    f = I.random_box_field(5, 19, 23, seed=71, lnk_var=2.0, n_wells=6, n_inactive=60, well_scale=4.0)
    cells, frac = I.explicit_particles(f, n, seed=n, active_only=False)
    ta = I.t_adv_of(f, 1e-4, 0.3)
    t0 = np.where(np.arange(n) % 3 == 0, 0.3 * ta, 0.0)   # a third starts at or after the first stop time
    state = dict(O.release_explicit(f, cells, frac), t=t0)
    with mp.Context(0) as ctx:
        fh = ctx.field(f)
        gh = ctx.release_explicit(fh, cells, frac, t0)
        for stop in (0.2 * ta, 0.3 * ta, np.inf):
            ref = O.track(f, state, t_stop=stop, arith="mirror")
            req = ctx.track(gh, t_stop=stop, flags=mp.TRACK_UPDATE_GROUP)
            ep = req.endpoints()
            req.free()
            for k in ("status", "cell", "px", "py", "pz", "t", "steps", "exit_face", "hash"):
                assert np.array_equal(ep[k], ref[k]), (k, stop)
            state = O.resume_state(ref)
        mp.mp_group_free(gh)
