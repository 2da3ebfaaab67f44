"""The FP64 recovery on meshes above the sizes where it takes the rows of R_M (recover_by_rows
in csrc/api.cu): h rows and momentum equations, against the oracle on a sample of the cells
and on the last ones (ragged blocks of 32: 3,528, 1,352 and 648 cells).
The smaller meshes of test_gpu_recover_fp64.py take the rows.

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


# the two sides of each line: by rows, by the momentum equations
@pytest.mark.parametrize("p,n", [(1, 128), (2, 40), (2, 42), (3, 24), (3, 26), (4, 16), (4, 18)])
@pytest.mark.parametrize("varying", [False, True])
def test_recovery_on_either_side_of_the_line(p, n, varying):
    from paper_2004_09389_gb300 import HDG_FP64, HDGSolver
    mesh = I.periodic_square_hierarchy(n, n_coarsest=4)
    rng = np.random.default_rng(p)
    f = rng.uniform(-1.0, 1.0, mesh.n_vertices) if varying else I.coriolis_flat(mesh, 1.0)
    tau, g, H = 8 * mesh.h, 1.3, 0.7
    prob = HDGProblem(mesh, p, tau=tau, g=g, H=H, f_vertex=f, lazy=True)
    ru = rng.standard_normal((mesh.n_cells, 2, prob.np))
    rh = rng.standard_normal((mesh.n_cells, prob.np))
    lam = rng.standard_normal((prob.n_facets, p + 1))
    s = HDGSolver(mesh, p, tau, g, H, f_vertex=f, precision=HDG_FP64)
    dev = [torch.from_numpy(a).cuda() for a in (ru, rh, lam)]
    u, h = torch.empty_like(dev[0]), torch.empty_like(dev[1])
    s.recover_dev(*dev, u, h)
    torch.cuda.synchronize()
    s.close()
    cells = np.unique(np.r_[np.arange(0, mesh.n_cells, 97), np.arange(mesh.n_cells - 40, mesh.n_cells)])
    q = prob.local_cells(cells, ru, rh, lam.ravel())
    uq, hq = q[:, :2 * prob.np], q[:, 2 * prob.np:]
    for a, b in ((u.cpu().numpy()[cells].reshape(len(cells), -1), uq), (h.cpu().numpy()[cells], hq)):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
