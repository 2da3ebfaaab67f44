"""Device memory of an FP64 handle: of R_M = A_K^-1 M_K it keeps the h rows and, only where f
varies over a cell, the three matrices of the velocity block (3 n_p^2 numbers per cell)
that the recovery reads."""
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


def test_velocity_block_only_where_f_varies():
    from paper_2004_09389_gb300 import HDG_FP64, HDGSolver
    mesh, p = I.periodic_square_hierarchy(192, n_coarsest=6), 3
    n_p = (p + 1) * (p + 2) // 2

    def taken(f):
        before = torch.cuda.mem_get_info()[0]
        s = HDGSolver(mesh, p, 8 * mesh.h, 1.0, 1.0, f_vertex=f, precision=HDG_FP64)
        torch.cuda.synchronize()
        after = torch.cuda.mem_get_info()[0]
        s.close()
        return before - after

    taken(np.ones(mesh.n_vertices))                      # the context and the module load first
    const = taken(np.ones(mesh.n_vertices))
    varying = taken(np.random.default_rng(0).uniform(-1.0, 1.0, mesh.n_vertices))
    block = 8 * mesh.n_cells * 3 * n_p ** 2
    assert abs(varying - const - block) <= 8 << 20       # allocations come in whole 2 MB pages
