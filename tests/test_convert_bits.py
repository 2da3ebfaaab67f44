"""The bitwise conversions between FP64, FP32 and float pairs (csrc/common.h) give the
plain conversions' results bit for bit: compiled with nvcc's host compiler and run on the
CPU.  Exact: no case may differ."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_conversions_are_exact(tmp_path):
    from paper_2004_09389_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = tmp_path / "convert_check"
    subprocess.run([nvcc, "-x", "cu", "-std=c++17", *build.ARCH, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "convert_check.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert int(out) == 0
