"""The automatic primal-dual schedule (footprint, launch count and halo chosen
by level size and iterations) against the explicit footprints: the same bits.

Sizes and counts lie where the rule changes footprint (one 32 x 16, 32 x 24,
32 x 32, 32 x 48, 64 x 24, 64 x 32, 64 x 48 or 64 x 64 per SM, two 64 x 32
per SM), at ragged edges and at the fewest iterations.  In 16-bit storage the
launch boundaries are part of the result: depth 8 up to 512 pixels, 6 above.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import f32pair, make_solver, np64

pytestmark = pytest.mark.gpu


def _run(pair, choice, iters, **prm):
    s = make_solver(pair, levels=1, **prm)
    s.set_schedule([choice])
    s.solve(pair["I0"], pair["I1"], 4, iters)
    out = [np64(s.read(0, b)) for b in ("U", "UBAR", "P")]
    s.close()
    return out


@pytest.mark.parametrize("W, H, iters", [
    (33, 21, 1), (33, 21, 2), (64, 64, 10), (64, 64, 30), (71, 130, 100), (160, 160, 20),
    (200, 200, 30), (256, 256, 100), (257, 333, 40), (400, 400, 10), (512, 512, 30),
    (640, 640, 10), (801, 600, 10), (1024, 768, 11)])
def test_automatic_schedule_equals_an_explicit_footprint(W, H, iters):
    p = f32pair(synth.plain_small(1, W=W, H=H, supersample=1))
    for prm in (dict(), dict(accel_gamma=0.3, precond=0)):
        for a, b in zip(_run(p, -1, iters, **prm), _run(p, 30, iters, **prm)):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("W, H, iters", [(64, 40, 17), (200, 200, 30), (513, 300, 13)])
def test_automatic_schedule_keeps_the_16_bit_rounding_points(W, H, iters, storage):
    p = f32pair(synth.plain_small(1, W=W, H=H, supersample=1))
    depth = 6 if W > 512 else 8                       # choice 24 + d: depth d on 64 x 64
    for a, b in zip(_run(p, -1, iters, storage=storage, pd_schedule=1),
                    _run(p, 24 + depth, iters, storage=storage, pd_schedule=1)):
        assert np.array_equal(a, b)
