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


@pytest.mark.gpu
@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("varying", [False, True])
def test_condensation_matches_oracle(p, varying):
    """Per-cell S_K of the FP64 condensation, both branches (f constant on every cell or
    not), on meshes whose cell count leaves a ragged last block (242 cells): 1e-12 of
    max |S_K|, the suite's tolerance for the FP64 operators."""
    import numpy as np
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import hdg_inputs as I
    from oracle.hdg import HDGProblem
    from paper_2004_09389_gb300 import HDGSolver, build
    build.build()
    mesh = I.periodic_square_hierarchy(11, n_coarsest=4)
    f = np.random.default_rng(0).uniform(-1.0, 1.0, mesh.n_vertices) if varying else I.coriolis_flat(mesh, 1.0)
    tau, g, H = 16 * mesh.h, 1.3, 0.7
    prob = HDGProblem(mesh, p, tau=tau, g=g, H=H, f_vertex=f)
    s = HDGSolver(mesh, p, tau, g, H, f_vertex=f)
    S, S0 = s.cell_schur(), np.stack([prob.cell_schur(K) for K in range(prob.N)])
    s.close()
    assert np.abs(S - S0).max() <= 1e-12 * np.abs(S0).max()
