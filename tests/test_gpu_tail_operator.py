"""The coarse cycle's tail as one dense product (csrc/k_p1.cu, dense_kernel): one
application of the preconditioner against the oracle's V-cycle, on hierarchies whose tails
take each rows-per-block variant and its remainders (first tail level of 100, 196, 576 and
784 vertices in FP64; the FP32 cycle of a handle whose levels do not merge in batches).

FP64 1e-12, FP32 1e-5 relative: the suite's tolerances for one preconditioner
application (the product adds n terms where the cycle summed about as many)."""
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


@pytest.mark.parametrize("n,n_coarsest", [(10, 5), (14, 7), (24, 3), (28, 7)])
def test_precond_with_dense_tail_matches_oracle(n, n_coarsest):
    from paper_2004_09389_gb300 import HDG_FP64, HDG_MIXED_FGMRES64, HDGSolver
    mesh = I.periodic_square_hierarchy(n, n_coarsest=n_coarsest)
    f = I.coriolis_flat(mesh, 1.0)
    tau, g, H = 8 * mesh.h / np.sqrt(1.3 * 0.7), 1.3, 0.7
    prob = HDGProblem(mesh, 1, tau=tau, g=g, H=H, f_vertex=f)
    pc = TwoLevelPreconditioner(prob, mesh, prob.trace_operator(), coarse="gmg")
    v = np.random.default_rng(n).standard_normal(prob.n_trace)
    z0 = pc(v)
    for precision, tol in ((HDG_FP64, 1e-12), (HDG_MIXED_FGMRES64, 1e-5)):
        s = HDGSolver(mesh, 1, tau, g, H, f_vertex=f, precision=precision)
        if precision == HDG_FP64:
            vd = torch.from_numpy(v).cuda()
            z = torch.empty_like(vd)
            s.precond_apply_dev(vd, z)
        else:
            vd = torch.from_numpy(v.astype(np.float32)).cuda()
            z = torch.empty_like(vd)
            s.precond_apply32_dev(vd, z)
        torch.cuda.synchronize()
        err = np.linalg.norm(z.cpu().numpy() - z0) / np.linalg.norm(z0)
        s.close()
        assert err <= tol
