"""A tuned schedule saved from one handle (fs_get_schedule) and set on another:
the same launches and, in 16-bit storage, where the results depend on them, the
same bits; there the tuner's choice is itself what the handle keeps."""
import numpy as np
import pytest

import synth
from gpu_helpers import f32pair, make_solver, np64

pytestmark = pytest.mark.gpu


def _frame(s, p):
    s.timing_enable(True)
    out = [np64(x) for x in s.solve(p["I0"], p["I1"], 3, 27)] + [np64(s.read(0, "P"))]
    return out, [n for _, n, _ in s.timing_read()]


@pytest.mark.parametrize("prm", [dict(), dict(precond=0, accel_gamma=0.3), dict(storage="f16"),
                                 dict(storage="bf16", pd_schedule=1), dict(regularizer="tgv")])
def test_a_saved_tuning_reproduces_the_handle_it_came_from(prm):
    p = f32pair(synth.plain_small(0))
    s1, s2, s3 = [make_solver(p, **prm) for _ in range(3)]
    assert s1.schedule() == [-1] * p["levels"]
    choice = s1.autotune(27)
    kept = s1.schedule()
    assert all(k in (-1, c) for k, c in zip(kept, choice))
    if "storage" in prm:
        assert kept == choice
    s2.set_schedule(kept)
    assert s2.schedule() == kept
    (a, na), (b, nb) = _frame(s1, p), _frame(s2, p)
    assert na == nb
    s3.set_schedule(choice)                 # the encoded choices: the same results
    for x, y, z in zip(a, b, _frame(s3, p)[0]):
        assert np.array_equal(x, y, equal_nan=True)
        assert np.array_equal(x, z, equal_nan=True)
    for s in (s1, s2, s3):
        s.close()


def test_persistent_handles_keep_the_choice():
    p = f32pair(synth.plain_small(0))
    s = make_solver(p, pd_schedule="persistent")
    assert s.autotune(20) == s.schedule()
    s.close()


@pytest.mark.parametrize("regularizer, last", [("huber_tv", 71), ("tgv", 40)])
def test_every_choice_reads_back(regularizer, last):
    p = f32pair(synth.plain_small(0, W=64, H=64, supersample=1))
    s = make_solver(p, levels=1, regularizer=regularizer)
    for c in range(-1, last + 1):
        s.set_schedule([c])
        assert s.schedule() == [c]
    s.close()
