"""Timing switched on between two batch solves on the same buffers: the graph
captured without the events has to be captured again."""
import pytest
import torch

from gpu_helpers import make_solver, ragged_pair

pytestmark = pytest.mark.gpu


def test_timing_enabled_after_a_batch_graph_was_captured():
    import paper_1909_07545_gb300 as fsb
    p = ragged_pair(3)
    ims = [torch.as_tensor(p[k], dtype=torch.float32, device="cuda") for k in ("I0", "I1")]
    out = torch.empty(2, *ims[0].shape, device="cuda")
    s = make_solver(p)
    b = fsb.Batch([s])
    for on in (False, True, False, True):
        s.timing_enable(on)
        b.solve([ims[0]], [ims[1]], 2, 10, disps=[out[0]], depths=[out[1]])
        times = s.timing_read(reset=True)
        assert all((ms > 0 and n > 0) if on else (ms == 0 and n == 0) for ms, n, _ in times)
    b.close()
    s.close()
