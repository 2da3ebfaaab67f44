"""The condensed right-hand side of FP64 handles (W_K of csrc/k_condense.cu) in its last
digits: smooth right-hand sides, p = 1..4, without rotation and with f varying over the
cells, Courant 16, on 242 cells, against long double.

Tolerance n_K 2^-52 relative: row of W_K times r_K is a sum of n_K products whose terms
hardly cancel for smooth data, each entry of W_K rounded once or twice (an FP64 solve with
one step of refinement)."""
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
@pytest.mark.parametrize("varying", [False, True])
def test_condensed_rhs_is_exact_to_rounding(p, varying):
    import extended
    from paper_2004_09389_gb300 import HDG_FP64, HDG_MIXED_FGMRES64, HDGSolver
    mesh = I.periodic_square_hierarchy(11, n_coarsest=4)
    f = np.random.default_rng(0).uniform(-1.0, 1.0, mesh.n_vertices) if varying else np.zeros(mesh.n_vertices)
    g, H = 1.3, 0.7
    tau = 16 * mesh.h / np.sqrt(g * H)
    prob = HDGProblem(mesh, p, tau=tau, g=g, H=H, f_vertex=f)
    x, y = np.moveaxis(I.dg_node_positions(mesh, p), -1, 0) * 2.0 * np.pi
    ru = np.stack([np.cos(x) + 0.4 * np.sin(2 * y + 0.3), np.sin(x + y) + 0.2], axis=1)
    rh = 1.0 + 0.3 * np.cos(2 * x - y)
    exact = extended.condensed_rhs(prob, ru, rh)
    for precision in (HDG_FP64, HDG_MIXED_FGMRES64):
        s = HDGSolver(mesh, p, tau, g, H, f_vertex=f, precision=precision)
        gd = torch.empty(prob.n_facets, p + 1, dtype=torch.float64, device="cuda")
        s.condensed_rhs_dev(torch.from_numpy(ru).cuda(), torch.from_numpy(rh).cuda(), gd)
        torch.cuda.synchronize()
        s.close()
        d = gd.cpu().numpy().ravel() - exact
        assert np.sqrt((d * d).sum()) <= 3 * prob.np * 2.0 ** -52 * np.sqrt((exact * exact).sum())


@pytest.mark.parametrize("p", [2, 3, 4])
def test_condensed_rhs_of_r_h_alone(p):
    """r_u = 0, f = 0: sums of n_p products of entries that are exact to their own rounding,
    (n_p + 2) 2^-53 relative (each product and addition rounds once, an entry twice)."""
    import extended
    from paper_2004_09389_gb300 import HDG_FP64, HDGSolver
    mesh = I.periodic_square_hierarchy(11, n_coarsest=4)
    f, g, H = np.zeros(mesh.n_vertices), 1.3, 0.7
    tau = 16 * mesh.h / np.sqrt(g * H)
    prob = HDGProblem(mesh, p, tau=tau, g=g, H=H, f_vertex=f)
    x, y = np.moveaxis(I.dg_node_positions(mesh, p), -1, 0) * 2.0 * np.pi
    rh = 0.2 + np.cos(2 * x - y) + 0.5 * np.sin(x + 0.4)
    ru = np.zeros((mesh.n_cells, 2, prob.np))
    exact = extended.condensed_rhs(prob, ru, rh)
    s = HDGSolver(mesh, p, tau, g, H, f_vertex=f, precision=HDG_FP64)
    gd = torch.empty(prob.n_facets, p + 1, dtype=torch.float64, device="cuda")
    s.condensed_rhs_dev(torch.from_numpy(ru).cuda(), torch.from_numpy(rh).cuda(), gd)
    torch.cuda.synchronize()
    s.close()
    d = gd.cpu().numpy().ravel() - exact
    assert np.sqrt((d * d).sum()) <= (prob.np + 2) * 2.0 ** -53 * np.sqrt((exact * exact).sum())
