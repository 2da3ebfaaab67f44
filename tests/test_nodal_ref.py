"""The nodal reference matrices (csrc/refelem.cpp, build_nodal_ref) equal the weak
ones multiplied by the inverse mass matrix, and the derivative entries that the
kernels leave out vanish: compiled with nvcc's host compiler and run on the CPU.
Entries are O(1) to O(p^2) sums of at most 15 terms: 1e-14 is about 50 ulp."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2004_09389_gb300", "csrc")


def test_nodal_matrices(tmp_path):
    from paper_2004_09389_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = tmp_path / "nodal_check"
    subprocess.run([nvcc, "-x", "cu", "-std=c++17", *build.ARCH, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "nodal_check.cpp"), os.path.join(CSRC, "refelem.cpp"), "-o", str(exe)],
                   check=True)
    worst, left_out = (float(v) for v in subprocess.run([str(exe)], check=True, capture_output=True,
                                                        text=True).stdout.split())
    assert worst <= 1e-14 and left_out <= 1e-14
