"""Copy waits of the TMA-staged footprints that run out: the CTA stays until
its own copies have landed, so a wait limit far below a copy's latency leaves
nothing behind that could write into another CTA's shared memory."""
import numpy as np
import pytest

import synth
from gpu_helpers import f32pair, make_solver, np64

pytestmark = pytest.mark.gpu

TMA = 55            # choice TMA + d = depth d on the TMA footprints


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_a_limit_below_a_copys_latency(storage):
    import paper_1909_07545_gb300 as fsb
    p = f32pair(synth.plain_small(0))
    args = (p["I0"], p["I1"], 3, 10)
    s = make_solver(p, storage=storage)
    s.set_schedule([TMA + 6, TMA + 4, -1])
    ref = [np64(x) for x in s.solve(*args)]
    s.check_waits()
    s.set_wait_limit(1e-9)
    for _ in range(5):
        s.solve(*args)
    try:
        s.check_waits()                # whether any copy was late is the clock's affair
    except fsb.FsError as e:
        assert e.status == -5          # FS_ETIMEOUT
    s.set_wait_limit(2.0)
    got = [np64(x) for x in s.solve(*args)]
    s.check_waits()
    for a, b in zip(got, ref):
        assert np.array_equal(a, b, equal_nan=True)
    s.close()
