"""Whole solves on levels whose automatic schedule takes the TMA-staged
footprints: buffer sets that change places with their tensor maps (odd numbers
of launches), chains of one or two launches a warp, a last warp with another
plan than the others, footprints left out outside a small FOV.  Against
explicit k_pd footprints: the same bits."""
import numpy as np
import pytest

from gpu_helpers import make_solver, np64

pytestmark = pytest.mark.gpu

BUFS = ("U", "UBAR", "UW", "P", "W")


def _pair(W, H, fov_px):
    """A level of W x H with an off-centre FOV circle of fov_px pixels' radius."""
    f = fov_px / np.radians(85.0)
    cam = dict(model="equidistant", fx=f, fy=f * 1.02, cx=0.47 * W + 0.3, cy=0.52 * H + 0.8, k=[0] * 4,
               fov_deg=170.0)
    y, x = np.mgrid[0:H, 0:W]
    rng = np.random.default_rng(W + H)
    im = lambda s: np.float32(0.5 + 0.3 * np.sin((x + s) / 5.0) * np.cos(y / 7.0) + 0.1 * rng.random((H, W)))
    return dict(I0=im(0.0), I1=im(0.4), cam0=cam, cam1=dict(cam), R=np.eye(3),
                t=np.array([-0.1, 0.0, 0.0]), levels=1, lam=50.0, eps=0.01)


def _tma_runs(p, iters, **prm):
    """Whether the level's schedule has TMA footprints: their waits run out."""
    import paper_1909_07545_gb300 as fsb
    s = make_solver(p, **prm)
    s.set_wait_limit(0.01)
    s.persist_stall(True)
    s.solve(p["I0"], p["I1"], 2, iters)
    try:
        s.check_waits()
        return False
    except fsb.FsError as e:
        assert e.status == -5
        return True
    finally:
        s.close()


# iters: one launch a warp, a chain of two, an odd number of more (and the even
# number the last of three warps has to take)
@pytest.mark.parametrize("prm", [dict(), dict(precond=0, accel_gamma=0.3), dict(use_graph=1)])
@pytest.mark.parametrize("warps", [1, 2, 3])
@pytest.mark.parametrize("iters", [5, 8, 13, 18, 24])
@pytest.mark.parametrize("W, H, fov_px", [(2048, 1701, 3000), (2251, 2048, 1000)])
def test_solves_equal_explicit_footprints(W, H, fov_px, iters, warps, prm):
    p = _pair(W, H, fov_px)
    outs = []
    for choice in (-1, 30):                           # 30: depth 6 on 64 x 64
        s = make_solver(p, **prm)
        s.set_schedule([choice])
        out = list(s.solve(p["I0"], p["I1"], warps, iters))
        out += [s.read(0, b) for b in BUFS]
        out += s.solve_continue(p["I1"], p["I0"], warps, iters)
        out += [s.read(0, b) for b in BUFS]
        s.check_waits()
        outs.append([np64(x) for x in out])
        s.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("W, H, fov_px", [(2048, 1701, 3000), (2251, 2048, 1000)])
def test_these_levels_run_the_tma_footprints(W, H, fov_px):
    p = _pair(W, H, fov_px)
    for iters in (8, 13, 18, 24) + ((5,) if fov_px == 1000 else ()):
        assert _tma_runs(p, iters), iters
