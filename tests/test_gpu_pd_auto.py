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


def _run(pair, choice, iters, bufs=("U", "UBAR", "P"), **prm):
    s = make_solver(pair, levels=1, **prm)
    s.set_schedule([choice])
    s.solve(pair["I0"], pair["I1"], 4, iters)
    out = [np64(s.read(0, b)) for b in bufs]
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


@pytest.mark.parametrize("prm", [dict(), dict(precond=0, accel_gamma=0.3), dict(storage="f16"),
                                 dict(storage="bf16", precond=0)])
@pytest.mark.parametrize("W, H, iters", [(1100, 900, 12), (1100, 900, 31)])
def test_footprints_outside_the_fov(W, H, iters, prm):
    # a small FOV circle off the image's centre: most footprints hold no FOV
    # pixel and are left out; the state outside the FOV, arbitrary here, still
    # ends with the bits of the footprint that treats every pixel
    cam = dict(model="equidistant", fx=120.0, fy=130.0, cx=400.3, cy=520.8, k=[0] * 4, fov_deg=170.0)
    rng = np.random.default_rng(5)
    p = dict(I0=rng.random((H, W)), I1=rng.random((H, W)), cam0=cam, cam1=dict(cam), R=np.eye(3),
             t=np.array([-0.1, 0.0, 0.0]), levels=1)
    state = {"U": rng.uniform(-1, 1, (H, W)), "UBAR": rng.uniform(-1, 1, (H, W)),
             "P": rng.uniform(-0.9, 0.9, (2, H, W))}
    outs = []
    for choice in (-1, 30):                           # 30: depth 6 on 64 x 64
        s = make_solver(p, levels=1, **prm)
        s.set_schedule([choice])
        s.solve(p["I0"], p["I1"], 1, 2)
        for b, v in state.items():
            s.write(0, b, v)
        s.stage(0, "PD", iters)
        outs.append([np64(s.read(0, b)) for b in state])
        s.solve(p["I0"], p["I1"], 2, iters)
        outs[-1] += [np64(s.read(0, b)) for b in state]
        s.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prm", [dict(), dict(precond=0, accel_gamma=0.3), dict(storage="f16"),
                                 dict(storage="bf16")])
@pytest.mark.parametrize("W, H, iters", [(2048, 1701, 13), (2251, 2048, 12)])
def test_large_levels_and_footprints_outside_the_fov(W, H, iters, prm):
    # the sizes at which the TMA-staged footprints are chosen, an off-centre
    # FOV, arbitrary state outside it
    cam = dict(model="equidistant", fx=450.0, fy=520.0, cx=900.3, cy=1020.8, k=[0] * 4, fov_deg=170.0)
    rng = np.random.default_rng(6)
    p = dict(I0=rng.random((H, W)), I1=rng.random((H, W)), cam0=cam, cam1=dict(cam), R=np.eye(3),
             t=np.array([-0.1, 0.0, 0.0]), levels=1)
    state = {"U": rng.uniform(-1, 1, (H, W)), "UBAR": rng.uniform(-1, 1, (H, W)),
             "P": rng.uniform(-0.9, 0.9, (2, H, W))}
    outs = []
    for choice in (-1, 30):
        s = make_solver(p, levels=1, **prm)
        s.set_schedule([choice])
        s.solve(p["I0"], p["I1"], 1, 2)
        for b, v in state.items():
            s.write(0, b, v)
        s.stage(0, "PD", iters)
        s.check_waits()
        outs.append([np64(s.read(0, b)) for b in state])
        s.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prm", [dict(), dict(precond=0, accel_gamma=0.3), dict(storage="f16")])
@pytest.mark.parametrize("warps, iters", [(1, 10), (2, 1), (3, 10), (4, 25), (5, 1)])
def test_odd_launch_counts(warps, iters, prm):
    # an odd number of launches leaves the state in the other buffer set: after
    # a frame of any number of warps, and one continued from it, all state is
    # where the explicit schedules (even counts, copies) leave it
    p = f32pair(synth.plain_small(1, W=133, H=70, supersample=1))
    outs = []
    for choice in (-1, 32):                           # 32: depth 8 on 64 x 64
        s = make_solver(p, levels=2, pd_schedule=1, **prm)
        s.set_schedule([choice, choice])
        s.timing_enable(True)
        out = list(s.solve(p["I0"], p["I1"], warps, iters))
        out += s.solve_continue(p["I1"], p["I0"], warps, iters)
        out += [s.read(l, b) for l in (0, 1) for b in ("U", "UBAR", "UW", "P", "W")]
        s.timing_read()
        outs.append([np64(x) for x in out])
        s.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b, equal_nan=True)


TGV = ("U", "UBAR", "V", "VBAR", "P", "Q")


@pytest.mark.parametrize("W, H, iters", [
    (33, 21, 1), (33, 21, 2), (50, 50, 100), (100, 90, 30), (200, 200, 100), (256, 256, 10),
    (401, 333, 30), (512, 512, 30), (900, 700, 11)])
def test_automatic_tgv_schedule_equals_a_launch_per_step(W, H, iters):
    p = f32pair(synth.plain_small(1, W=W, H=H, supersample=1))
    for a, b in zip(_run(p, -1, iters, TGV, regularizer="tgv"),
                    _run(p, 0, iters, TGV, regularizer="tgv")):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prm", [dict(), dict(precond=0, theta=0.5)])
@pytest.mark.parametrize("W, H, iters", [(1100, 900, 12), (700, 1100, 31)])
def test_tgv_footprints_outside_the_fov(W, H, iters, prm):
    # as above: state at rest and not at rest outside a small FOV circle
    cam = dict(model="equidistant", fx=120.0, fy=130.0, cx=400.3, cy=520.8, k=[0] * 4, fov_deg=170.0)
    rng = np.random.default_rng(6)
    p = dict(I0=rng.random((H, W)), I1=rng.random((H, W)), cam0=cam, cam1=dict(cam), R=np.eye(3),
             t=np.array([-0.1, 0.0, 0.0]), levels=1)
    shape = dict(U=(H, W), UBAR=(H, W), V=(2, H, W), VBAR=(2, H, W), P=(2, H, W), Q=(4, H, W))
    state = {b: rng.uniform(-1.5, 1.5, shape[b]) for b in TGV}
    outs = []
    for choice in (-1, 0):
        s = make_solver(p, levels=1, regularizer="tgv", **prm)
        s.set_schedule([choice])
        s.solve(p["I0"], p["I1"], 1, 2)
        M = np64(s.read(0, "MASK")) > 0.5
        for b, v in state.items():
            s.write(0, b, v)
        s.stage(0, "PD", iters)
        # (a launch per step leaves the pixels outside the FOV as they are)
        outs.append([np64(s.read(0, b))[..., M] for b in TGV])
        s.solve(p["I0"], p["I1"], 2, iters)
        outs[-1] += [np64(s.read(0, b)) for b in TGV]
        s.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
