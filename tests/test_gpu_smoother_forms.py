"""The two forms of the facet sweeps (csrc/k_trace.cu): on the rows of D^-1 S (FP64 handles;
FP32 where hat_pays32 in csrc/api.cu takes them) and on those of S with the inverse blocks
(FP32 in the band of sizes between; the FP64 cycle of a mixed handle).  One preconditioner
application in each, on both sides of the band, against the FP64 cycle of the same handle,
and the two FP64 forms against each other.

1e-5 relative in FP32 and 1e-12 in FP64: the suite's tolerances for one application."""
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


@pytest.mark.parametrize("smoother", [0, 1])
@pytest.mark.parametrize("n,p", [(13, 1), (64, 2), (160, 3), (192, 4), (256, 4)])
def test_forms_agree(n, p, smoother):
    from paper_2004_09389_gb300 import HDG_FP64, HDG_MIXED_FP32, HDGSolver
    mesh = I.periodic_square_hierarchy(n, n_coarsest=4 if n % 4 == 0 else 13)
    f = I.coriolis_flat(mesh, 1.0)
    tau, g, H = 8 * mesh.h / np.sqrt(1.3 * 0.7), 1.3, 0.7
    more = {"smoother": smoother, **({"cheb_theta": 1.15, "cheb_delta2": 0.3} if smoother else {})}
    z = {}
    for precision in (HDG_FP64, HDG_MIXED_FP32):
        s = HDGSolver(mesh, p, tau, g, H, f_vertex=f, precision=precision, **more)
        v = torch.from_numpy(np.random.default_rng(n).standard_normal(s.n_trace).astype(np.float32)).cuda()
        z[precision] = torch.empty(s.n_trace, dtype=torch.float64, device="cuda")
        s.precond_apply_dev(v.double(), z[precision])
        if precision == HDG_MIXED_FP32:
            z32 = torch.empty_like(v)
            s.precond_apply32_dev(v, z32)
        torch.cuda.synchronize()
        s.close()
    ref = z[HDG_FP64]
    assert float((z[HDG_MIXED_FP32] - ref).norm() / ref.norm()) <= 1e-12
    assert float((z32.double() - ref).norm() / ref.norm()) <= 1e-5
