"""The two-float cell solve (step 1 of the mixed handles, csrc/k_ff.cu): the condensed
right-hand side and the recovery from explicit inputs against the oracle, with f constant
on every cell and varying over the cells (two kernels each), p = 1..4, on a mesh whose
cell count (242) leaves a ragged last tile of 32 cells.

1e-12 relative, the suite's tolerance for the two-float steps: about 2^-47 per operation,
times the weak gradient's norm (tau c |G| of order Courant x p^2, 128 at most here)."""
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


def _rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b))


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("varying", [False, True])
def test_rhs_and_recovery_match_oracle(p, varying):
    from paper_2004_09389_gb300 import HDG_MIXED_FP32, HDGSolver
    mesh = I.periodic_square_hierarchy(11, n_coarsest=4)
    rng = np.random.default_rng(p)
    f = rng.uniform(-1.0, 1.0, mesh.n_vertices) if varying else I.coriolis_flat(mesh, 1.0)
    tau, g, H = 8 * mesh.h, 1.3, 0.7
    prob = HDGProblem(mesh, p, tau=tau, g=g, H=H, f_vertex=f)
    ru = rng.standard_normal((mesh.n_cells, 2, prob.np))
    rh = rng.standard_normal((mesh.n_cells, prob.np))
    lam = rng.standard_normal((prob.n_facets, p + 1))
    s = HDGSolver(mesh, p, tau, g, H, f_vertex=f, precision=HDG_MIXED_FP32)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (ru, rh, lam)]
    gd, u, h = torch.empty_like(dev[2]), torch.empty_like(dev[0]), torch.empty_like(dev[1])
    s.condensed_rhs_dev(dev[0], dev[1], gd)
    s.recover_dev(dev[0], dev[1], dev[2], u, h)
    torch.cuda.synchronize()
    u0, h0 = prob.recover(lam.ravel(), ru, rh)
    assert _rel(gd.cpu().numpy(), prob.condensed_rhs(ru, rh)) <= 1e-12
    assert _rel(u.cpu().numpy(), u0) <= 1e-12 and _rel(h.cpu().numpy(), h0) <= 1e-12
    s.close()
