"""The FP64 recovery (csrc/k_trace.cu): h by the rows of R_M and X_B, the velocity from the
momentum equations, against the oracle, p = 1..4, without rotation, with f constant on
every cell and varying, on a mesh whose cell count (242) leaves a ragged block of 32 cells.

1e-12 relative, the suite's tolerance for the FP64 steps."""
import numpy as np
import pytest

import hdg_inputs as I
from oracle.hdg import HDGProblem

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_09389_gb300 import build
    build.build()


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("f0", [0.0, 1.0, "varying"])
def test_recovery_matches_oracle(p, f0):
    from paper_2004_09389_gb300 import HDG_FP64, HDG_MIXED_FGMRES64, HDGSolver
    mesh = I.periodic_square_hierarchy(11, n_coarsest=4)
    rng = np.random.default_rng(p)
    f = rng.uniform(-1.0, 1.0, mesh.n_vertices) if f0 == "varying" else I.coriolis_flat(mesh, f0)
    tau, g, H = 12 * mesh.h, 1.3, 0.7
    prob = HDGProblem(mesh, p, tau=tau, g=g, H=H, f_vertex=f)
    ru = rng.standard_normal((mesh.n_cells, 2, prob.np))
    rh = rng.standard_normal((mesh.n_cells, prob.np))
    lam = rng.standard_normal((prob.n_facets, p + 1))
    u0, h0 = prob.recover(lam.ravel(), ru, rh)
    for precision in (HDG_FP64, HDG_MIXED_FGMRES64):
        s = HDGSolver(mesh, p, tau, g, H, f_vertex=f, precision=precision)
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (ru, rh, lam)]
        u, h = torch.empty_like(dev[0]), torch.empty_like(dev[1])
        s.recover_dev(dev[0], dev[1], dev[2], u, h)
        torch.cuda.synchronize()
        s.close()
        for a, b in ((u, u0), (h, h0)):
            assert np.linalg.norm(a.cpu().numpy().ravel() - np.ravel(b)) <= 1e-12 * np.linalg.norm(np.ravel(b))
