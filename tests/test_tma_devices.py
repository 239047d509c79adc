"""The TMA-staged footprints on every device of a process (no GPU: the host
code of the launch runs against a fake CUDA runtime of two devices)."""
import os
import shutil
import subprocess

import pytest

from paper_1909_07545_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_each_device_is_opted_in_and_gets_its_own_grid(tmp_path):
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None or not shutil.which(build.nvcc()):
        pytest.skip("no compiler")
    build.build()
    fake, exe = tmp_path / "fake_cudart.o", tmp_path / "check"
    objs = [os.path.join(build.BUILD, o) for o in ("k_pd_tma.o", "k_pd.o")]
    for cmd in ([cc, "-c", os.path.join(ROOT, "tests", "fake_cudart.c"), "-o", str(fake)],
                [build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-cudart", "none",
                 "-I", build.INCLUDE, "-I", build.CSRC,
                 os.path.join(ROOT, "tests", "tma_devices_check.cu"), *objs, str(fake), "-o", str(exe)]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
