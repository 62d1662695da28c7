"""The float64 digit products' host logic (csrc/f64_digits.cu) with a stand-in
for the CUDA runtime: after a step that failed or was not checked, the next run
starts from cleared sums."""
import os
import subprocess

import pytest

from paper_1101_0265_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_sums_are_cleared_after_a_failed_step(tmp_path):
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "f64_state")
    cmd = [cc, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-cudart", "none", "-I", os.path.join(build.ROOT, "include"),
           "-I", build.CSRC, os.path.join(build.CSRC, "f64_digits.cu"), os.path.join(HERE, "native", "f64_state.cc"),
           "-o", exe] + build.ARCH
    p = subprocess.run(cmd, capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    p = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout
