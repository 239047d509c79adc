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


def test_served_request_whose_copy_wait_runs_out_fails(monkeypatch):
    # a level large enough for the automatic schedule to take the TMA footprints;
    # the rig's next frame, on a fresh handle, gives a lone handle's bits
    import paper_1909_07545_gb300 as fsb
    W, H = 1400, 1360
    rng = np.random.default_rng(3)
    cam = dict(model="equidistant", fx=460.0, fy=460.0, cx=(W - 1) / 2, cy=(H - 1) / 2, k=[0] * 4,
               fov_deg=170.0)
    p = dict(I0=np.float32(rng.random((H, W))), I1=np.float32(rng.random((H, W))), cam0=cam,
             cam1=dict(cam), R=np.eye(3), t=np.array([-0.1, 0.0, 0.0]), levels=1)
    srv = fsb.Server(warps=1, iters=16, cold_warps=2, cold_iters=16, autotune=0)
    rig = srv.add_rig(cam, dict(cam), p["R"], p["t"], W, H, 1)
    out = [np.empty((H, W), np.float32) for _ in range(2)]
    monkeypatch.setenv("FS_FAULT_WAIT", "0.02")
    for _ in range(2):                     # cold both times: no result to continue from
        req = srv.submit(rig, p["I0"], p["I1"], *out)
        with pytest.raises(fsb.FsError, match="copy wait") as e:
            srv.wait(req)
        assert e.value.status == -3        # FS_ECUDA
    st = srv.stats()
    assert st["failed"] == 2 and st["cold"] == 2
    monkeypatch.delenv("FS_FAULT_WAIT")
    srv.evict_all()
    for _ in range(2):                     # cold, then continued
        srv.wait(srv.submit(rig, p["I0"], p["I1"], *out))
    srv.close()
    s = make_solver(p, lam=50.0, huber_eps=0.01)
    s.solve(p["I0"], p["I1"], 2, 16)
    ref = [np64(x) for x in s.solve_continue(p["I0"], p["I1"], 1, 16)]
    s.check_waits()
    s.close()
    for a, b in zip(out, ref):
        assert np.array_equal(a, b, equal_nan=True)
