"""The reciprocal square root of the ball projections, over every non-negative
float: the flushing form gives the bits of rsqrtf wherever it is used."""
import os
import subprocess

import pytest

from paper_1909_07545_gb300 import build

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_flushing_form_equals_rsqrtf_on_every_float(tmp_path):
    exe = str(tmp_path / "check")
    r = subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", build.INCLUDE, "-I", build.CSRC,
                        os.path.join(ROOT, "tests", "ball_scale_check.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.split() == ["0", "0"], r.stdout + r.stderr
