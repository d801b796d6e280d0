"""Double-float arithmetic of the Gaussian draws on the CPU (tests/ddmath_check.cu): radii within 4e-13, cosines and sines within
1e-13, a quarter of what the rounding test of a draw allows for."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_errors(tmp_path):
    from paper_2404_07249_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "ddmath_check")
    r = subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-O1", "-Xcompiler", "-ffp-contract=off", "-I", build.CSRC,
                        os.path.join(ROOT, "tests", "ddmath_check.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
