"""Forms of one kernel that meet in one call or follow each other without a wait.

* A merged batch whose problems take different forms (FP32 sweeps on S beside sweeps on
  D^-1 S, f constant beside varying, single-CTA tails beside dense ones): the same bits as
  each problem alone.
* set_tau directly behind a solve and a recovery that nothing has waited for (the coarse
  operators are rebuilt on the handle's side stream meanwhile): the same bits as with a
  wait after every call."""
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


def _rhs(mesh, p, seed):
    rng = np.random.default_rng(seed)
    n_p = (p + 1) * (p + 2) // 2
    return (torch.from_numpy(rng.standard_normal((mesh.n_cells, 2, n_p))).cuda(),
            torch.from_numpy(rng.standard_normal((mesh.n_cells, n_p))).cuda())


def test_batch_of_different_forms():
    from paper_2004_09389_gb300 import HDG_MIXED_FP32, HDGSolver, MergedBatch
    # 49,152 facets at p = 3: the size where FP32 sweeps take S; 16 x 16 coarsest levels alone: dense tails
    solvers, ru, rh = [], [], []
    for k, (kind, size, p, coarsest) in enumerate([("flat", 128, 3, 4), ("flat", 32, 3, 4), ("sphere", 3, 3, 1),
                                                   ("flat", 16, 1, 16), ("flat", 48, 2, 24)]):
        if kind == "flat":
            mesh = I.periodic_square_hierarchy(size, n_coarsest=coarsest)
            f = I.coriolis_flat(mesh, 1.0)
        else:
            mesh = I.sphere_hierarchy(size, 1.0, r_coarsest=coarsest)
            f = I.coriolis_sphere(mesh, 0.5)
        solvers.append(HDGSolver(mesh, p, 4.0 * mesh.h, 1.0, 1.0, f_vertex=f, rtol=1e-10, precision=HDG_MIXED_FP32))
        a, b = _rhs(mesh, p, k)
        ru.append(a)
        rh.append(b)
    alone = [torch.empty((s.n_facets, s.p + 1), dtype=torch.float64, device="cuda") for s in solvers]
    for s, a, b, lam in zip(solvers, ru, rh, alone):
        s.solve_dev(a, b, lam)
    batch = MergedBatch(solvers)
    lam = [torch.empty_like(x) for x in alone]
    batch.solve_dev(ru, rh, lam)
    torch.cuda.synchronize()
    for i, (x, y) in enumerate(zip(lam, alone)):
        assert torch.equal(x, y), i
    batch.close()
    for s in solvers:
        s.close()


@pytest.mark.parametrize("precision", ["HDG_FP64", "HDG_MIXED_FP32"])
def test_set_tau_behind_a_running_solve(precision):
    import paper_2004_09389_gb300 as lib
    mesh, p = I.sphere_hierarchy(4, 1.0, r_coarsest=1), 2
    tau = 4.0 * mesh.h
    s = lib.HDGSolver(mesh, p, tau, 1.0, 1.0, f_vertex=I.coriolis_sphere(mesh, 0.5), rtol=1e-10,
                      precision=getattr(lib, precision))
    ru, rh = _rhs(mesh, p, 7)
    kept = precision == "HDG_MIXED_FP32"

    def loop(wait):
        out = []
        for scale in (1.0, 0.5, 2.0, 1.0):
            s.set_tau(scale * tau)
            lam = torch.empty((s.n_facets, p + 1), dtype=torch.float64, device="cuda")
            u, h = torch.empty_like(ru), torch.empty_like(rh)
            s.solve_dev(ru, rh, lam)
            s.recover_dev(*((None, None) if kept else (ru, rh)), None, u, h)
            if wait:
                torch.cuda.synchronize()
            out += [lam, u, h]
        torch.cuda.synchronize()
        return out

    for x, y in zip(loop(False), loop(True)):
        assert torch.equal(x, y)
    s.close()
