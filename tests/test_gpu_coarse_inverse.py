"""The inverse of the coarsest P1 level (csrc/k_condense.cu): one application of the
preconditioner against the oracle's V-cycle with 9 and 144 coarsest vertices (in-place in
shared memory), 169 (one block over global memory) and 289 (two launches per column), and
the P1 levels assembled in one launch, with and without rotation.

1e-12 relative: the suite's tolerance for one FP64 preconditioner application."""
import numpy as np
import pytest

import hdg_inputs as I
from oracle.hdg import HDGProblem
from oracle.solver import TwoLevelPreconditioner

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_09389_gb300 import build
    build.build()


@pytest.mark.parametrize("n_coarsest", [3, 12, 13, 17])
@pytest.mark.parametrize("f0", [0.0, 1.0])
def test_precond_matches_oracle(n_coarsest, f0):
    from paper_2004_09389_gb300 import HDGSolver
    mesh = I.periodic_square_hierarchy(2 * n_coarsest, n_coarsest=n_coarsest)
    f = I.coriolis_flat(mesh, f0)
    tau, g, H = 8 * mesh.h / np.sqrt(1.3 * 0.7), 1.3, 0.7
    prob = HDGProblem(mesh, 2, tau=tau, g=g, H=H, f_vertex=f)
    pc = TwoLevelPreconditioner(prob, mesh, prob.trace_operator(), coarse="gmg")
    v = np.random.default_rng(n_coarsest).standard_normal(prob.n_trace)
    s = HDGSolver(mesh, 2, tau, g, H, f_vertex=f)
    vd = torch.from_numpy(v).cuda()
    z = torch.empty_like(vd)
    s.precond_apply_dev(vd, z)
    torch.cuda.synchronize()
    s.close()
    z0 = pc(v)
    assert np.linalg.norm(z.cpu().numpy() - z0) <= 1e-12 * np.linalg.norm(z0)
