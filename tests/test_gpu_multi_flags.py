"""A batched call reports a wait that gave up in any of its fields, not only in the last one of a context: a program that
stands in for the library's step after each contraction and raises the context's error flag there (no wait is made to run
out)."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_flag_of_any_field(tmp_path):
    from paper_2404_07249_gb300 import build
    lib = build.build()
    exe = str(tmp_path / "multi_flags_check")
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", build.CSRC,
                        os.path.join(ROOT, "tests", "multi_flags_check.cu"), "-o", exe, "-Xlinker", "--export-dynamic",
                        "-L", os.path.dirname(lib), "-lpolybin", "-ldl", "-Xlinker", "-rpath," + os.path.dirname(lib)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:]
    assert r.stdout.strip().endswith("0 failures")
