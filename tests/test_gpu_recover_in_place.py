"""The recovery writes a cell's (u, h) after it has read that cell's right-hand side, so the
outputs may be the right-hand side's own buffers: the same bits as with buffers of their own,
for the rows (small meshes, p = 1), the momentum form and the two-float form."""
import numpy as np
import pytest

import hdg_inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_09389_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["HDG_FP64", "HDG_MIXED_FP32"])
@pytest.mark.parametrize("p,n", [(1, 64), (2, 38), (2, 42), (3, 22), (3, 26), (4, 14), (4, 18)])
def test_outputs_in_the_right_hand_sides_buffers(p, n, precision):
    import paper_2004_09389_gb300 as lib
    mesh = I.periodic_square_hierarchy(n, n_coarsest=4)
    rng = np.random.default_rng(n)
    n_p = (p + 1) * (p + 2) // 2
    s = lib.HDGSolver(mesh, p, 8 * mesh.h, 1.3, 0.7, f_vertex=I.coriolis_flat(mesh, 1.0),
                      precision=getattr(lib, precision))
    ru = torch.from_numpy(rng.standard_normal((mesh.n_cells, 2, n_p))).cuda()
    rh = torch.from_numpy(rng.standard_normal((mesh.n_cells, n_p))).cuda()
    lam = torch.from_numpy(rng.standard_normal((s.n_facets, p + 1))).cuda()
    u, h = torch.empty_like(ru), torch.empty_like(rh)
    s.recover_dev(ru, rh, lam, u, h)
    s.recover_dev(ru, rh, lam, ru, rh)
    torch.cuda.synchronize()
    assert torch.equal(u, ru) and torch.equal(h, rh)
    s.close()
