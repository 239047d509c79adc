"""A pose change of a batch's handle between two calls on the same buffers: the
batch's graph holds the depth's constants, so it has to be captured again."""
import numpy as np
import pytest
import torch

from gpu_helpers import make_solver, np64, ragged_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sched", ["auto", "persistent"])
def test_batch_after_set_pose_equals_the_handle_alone(sched):
    import paper_1909_07545_gb300 as fsb
    p = ragged_pair(3)
    ims = [torch.as_tensor(p[k], dtype=torch.float32, device="cuda") for k in ("I0", "I1")]
    out = torch.empty(2, *ims[0].shape, device="cuda")
    s = make_solver(p, pd_schedule=sched)
    b = fsb.Batch([s])
    for t in (p["t"], 2.0 * p["t"], p["t"]):        # the same directions, another baseline
        s.set_pose(p["R"], t)
        b.solve([ims[0]], [ims[1]], 2, 10, disps=[out[0]], depths=[out[1]])
        got = np64(out)
        ref = make_solver(dict(p, t=t))
        d, z = ref.solve(*ims, 2, 10)
        assert np.array_equal(got[0], np64(d))
        assert np.array_equal(got[1], np64(z), equal_nan=True)
        ref.close()
    b.close()
    s.close()
