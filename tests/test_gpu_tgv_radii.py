"""The ball projections of the TGV dual step, by the radii alpha1 and alpha0:
radii of 1e-18 and more take the flushing reciprocal square root in the
blocked kernel, smaller ones the full-range one.  The launch-per-step
kernels (schedule 0) always take the full-range one; every choice has to
give their bits."""
import numpy as np
import pytest

import synth
from gpu_helpers import f32pair, make_solver, np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha0, alpha1", [(17.0, 1.2), (0.0, 1.2), (1e-18, 1e-18),
                                            (1e-20, 1.2), (1e-21, 1e-21)])
def test_blocked_projection_equals_the_stepwise_one(alpha0, alpha1):
    p = f32pair(synth.plain_small(0, W=96, H=72))
    outs = []
    for choice in (0, 4, 12, 36):            # per step; 4, 1 and 2 rows a thread
        s = make_solver(p, levels=1, regularizer="tgv", alpha0=alpha0, alpha1=alpha1)
        s.set_schedule([choice])
        s.solve(p["I0"], p["I1"], 2, 9)
        outs.append([np64(s.read(0, b)) for b in ("U", "P", "V", "Q")])
        s.close()
    assert np.isfinite(outs[0][0]).all()
    for o in outs[1:]:
        for a, b in zip(o, outs[0]):
            assert np.array_equal(a, b)
