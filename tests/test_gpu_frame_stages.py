"""A solve (level starts and frame ends in one launch each) against the same
frame stage by stage: the same bits, from zero, from a given disparity and
continued, at ragged sizes and with every kind of constants a warp start writes.
"""
import numpy as np
import pytest

from gpu_helpers import f32pair, make_solver, np64, ragged_pair

pytestmark = pytest.mark.gpu

WARPS, ITERS, LEVELS = 2, 7, 2


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("W, H, levels", [(203, 157, 6), (17, 40, 3), (64, 41, 2), (15, 16, 1),
                                          (393, 385, 5), (401, 400, 5)])
def test_pyramid_equals_its_stages(W, H, levels, storage):
    # both sides of the size rule, ragged edges, more levels than one launch makes
    p = f32pair(ragged_pair(4, W=W, H=H))
    outs = []
    for stages in (False, True):
        s = make_solver(p, levels=levels, storage=storage)
        if stages:
            s.write(0, "I0", p["I0"])
            s.prerotate(p["I1"])
            for l in range(levels - 1):
                s.stage(l, "DOWNSAMPLE")
        else:
            s.solve(p["I0"], p["I1"], 1, 1)
        outs.append([np64(s.read(l, b)) for l in range(levels) for b in ("I0", "I1")])
        s.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


def _warps(s, level):
    s.stage(level, "WARP")
    for w in range(WARPS):
        s.stage(level, "PD", ITERS)
        s.stage(level, "CLIP_WARP" if w + 1 < WARPS else "CLIP")


def _by_stages(s, p, how, init, tgv):
    s.write(0, "I0", p["I0"])
    s.prerotate(p["I1"])
    if how == "continue":          # u and w as they are, duals and v at zero
        s.write(0, "P", 0 * np64(s.read(0, "P")))
    elif how == "warm":
        s.write(0, "U", init)
        s.stage(0, "WARM")
    else:
        for l in range(LEVELS - 1):
            s.stage(l, "DOWNSAMPLE")
        for b in ("U", "W", "P"):
            s.write(LEVELS - 1, b, 0 * np64(s.read(LEVELS - 1, b)))
    for l in range(LEVELS - 1 if how == "cold" else 0, -1, -1):
        s.stage(l, "TENSOR")
        if how == "cold" and l + 1 < LEVELS:
            s.stage(l, "UPSAMPLE")
        elif tgv and how != "warm":
            for b in ("V", "Q"):
                s.write(l, b, 0 * np64(s.read(l, b)))
        _warps(s, l)
    return s.depth()


@pytest.mark.parametrize("prm", [
    dict(), dict(precond=0, deriv="central"), dict(storage="f16"), dict(storage="bf16"),
    dict(regularizer="tgv"), dict(regularizer="tgv", precond=0)], ids=str)
@pytest.mark.parametrize("how", ["cold", "warm", "continue"])
@pytest.mark.parametrize("W, H", [(203, 157), (64, 41)])
def test_solve_equals_its_stages(W, H, how, prm):
    p = f32pair(ragged_pair(3, W=W, H=H))
    init = np.random.default_rng(2).uniform(-1, 1, (H, W)).astype(np.float32)
    init[3, 5] = np.inf
    outs = []
    for stages in (False, True):
        s = make_solver(p, levels=LEVELS, pd_schedule=1, **prm)
        if how == "continue":
            s.solve(p["I0"], p["I1"], WARPS, ITERS)
        if stages:
            d = _by_stages(s, p, how, init, prm.get("regularizer") == "tgv")
        elif how == "continue":
            d = s.solve_continue(p["I0"], p["I1"], WARPS, ITERS)
        else:
            d = s.solve(p["I0"], p["I1"], WARPS, ITERS, init=init if how == "warm" else None)
        outs.append([np64(x) for x in d] + [np64(s.read(0, b)) for b in ("U", "W", "UW", "P")])
        s.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b, equal_nan=True)
