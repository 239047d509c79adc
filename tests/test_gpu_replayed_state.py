"""The stage interface after a replayed graph: a replay rewrites the levels'
step sizes and linearisation like the launches it was captured from, so the
iterations' stored constants have to be made again from what it left -- the
bits of a handle that launches every solve."""
import pytest
import torch

import synth
from gpu_helpers import f32pair, make_solver, np64

pytestmark = pytest.mark.gpu


def _images(seed):
    p = f32pair(synth.plain_small(seed, W=96, H=80, supersample=1))
    return p, [torch.as_tensor(p[k], dtype=torch.float32, device="cuda") for k in ("I0", "I1")]


def _run(graph, batch, stages, bufs, **prm):
    """solve, stage WARP, the same call on other images in the same buffers
    (with graph: a replay), then `stages`; the levels' state."""
    import paper_1909_07545_gb300 as fsb
    p, ims = _images(1)
    others = _images(2)[1]
    s = make_solver(p, levels=2, use_graph=int(graph), **prm)
    out = torch.empty(2, *ims[0].shape, device="cuda")
    b = fsb.Batch([s]) if batch and graph else None

    def solve():
        if b:
            b.solve([ims[0]], [ims[1]], 2, 10, disps=[out[0]], depths=[out[1]])
        else:
            s.solve(*ims, 2, 10, disp=out[0], depth=out[1])
    solve()
    for l in (0, 1):
        s.stage(l, "WARP")
    for a, o in zip(ims, others):
        a.copy_(o)
    solve()
    for l in (0, 1):
        for st, n in stages:
            s.stage(l, st, n)
    got = [np64(s.read(l, x)) for l in (0, 1) for x in bufs]
    if b:
        b.close()
    s.close()
    return got


HUBER, TGV = ("U", "UBAR", "P"), ("U", "UBAR", "V", "VBAR", "P", "Q")


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("prm, bufs", [
    (dict(), HUBER), (dict(storage="f16", pd_schedule=1), HUBER),
    (dict(pd_schedule="persistent"), HUBER), (dict(regularizer="tgv"), TGV)])
@pytest.mark.parametrize("stages", [[("PD", 12)], [("CLIP_WARP", 0), ("PD", 12)]])
def test_stages_after_a_replay(stages, prm, bufs, batch):
    for a, b in zip(_run(True, batch, stages, bufs, **prm), _run(False, batch, stages, bufs, **prm)):
        assert (a == b).all()
