"""The library's reference matrices (csrc/refelem.cpp) against exact rational arithmetic:
every entry is the exact value rounded to FP64, up to what the extended precision of the
quadrature and of M^-1 leaves.  The nodal matrices multiply the weak ones by M^-1, so
FP64 quadrature shows up in them several ulp large.

Tolerance 2^-52 of a matrix's largest entry: half of it for the rounding to FP64, the other
half covers 2^-64 (x86) times cond(M) <= 1e3 with a margin of 2."""
import os
import subprocess

import numpy as np
import pytest

from oracle import reference as ref

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2004_09389_gb300", "csrc")


@pytest.fixture(scope="module")
def dumped(tmp_path_factory):
    from paper_2004_09389_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = tmp_path_factory.mktemp("ref") / "reference_dump"
    subprocess.run([nvcc, "-x", "cu", "-std=c++17", *build.ARCH, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "reference_dump.cpp"), os.path.join(CSRC, "refelem.cpp"),
                    "-o", str(exe)], check=True)
    text = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [np.array([float.fromhex(v) for v in line.split()]) for line in text.splitlines()]


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_entries_are_the_exact_values_rounded_once(p, dumped, monkeypatch):
    monkeypatch.setattr(ref, "_f", lambda x: np.array(x, dtype=object))      # keep the Fractions
    R = ref.reference_matrices.__wrapped__(p)
    Mi = np.array(ref.exact_inverse(R["M"].tolist()), dtype=object)
    want = [R["M1"], *R["N"], Mi @ R["Dxi"], Mi @ R["Deta"], *(Mi @ N for N in R["N"]), Mi @ R["ML"][1],
            Mi @ R["ML"][2], -Mi @ R["Dxi"].T, -Mi @ R["Deta"].T]
    got, at = dumped[p - 1], 0
    for k, A in enumerate(want):
        b = got[at:at + A.size]
        at += A.size
        err = max(abs(float(x - ref.Fraction(y))) for x, y in zip(A.ravel(), b))
        assert err <= 2.0 ** -52 * max(abs(float(x)) for x in A.ravel()), (k, err)
    assert at == got.size
