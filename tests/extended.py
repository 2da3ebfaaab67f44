"""The condensed right-hand side (step 1) in extended precision, for tests of the FP64
steps' last digits: the cell systems of oracle/hdg.py from the exact rational reference
matrices, formed and solved in numpy's long double."""
import numpy as np

from oracle import reference as ref

LD = np.longdouble


def _ld(x):
    """Fractions to long double, rounded from an FP64 pair."""
    x = np.array(x, dtype=object)
    hi = x.astype(np.float64)
    lo = np.vectorize(lambda q, v: float(q - ref.Fraction(float(v))), otypes=[float])(x, hi)
    return hi.astype(LD) + lo.astype(LD)


def reference_matrices(p):
    keep, ref._f = ref._f, _ld
    try:
        R = ref.reference_matrices.__wrapped__(p)
    finally:
        ref._f = keep
    return R


def solve(A, b):
    """x = A^-1 b for the matrices [N][n][n] and vectors [N][n], elimination with partial pivoting."""
    A, b, idx, n = A.copy(), b.copy(), np.arange(len(A)), A.shape[1]
    for k in range(n):
        piv = k + np.abs(A[:, k:, k]).argmax(1)
        for M in (A, b):
            t = M[idx, piv].copy()
            M[idx, piv] = M[:, k]
            M[:, k] = t
        f = A[:, k + 1:, k] / A[:, k, k][:, None]
        A[:, k + 1:] -= f[..., None] * A[:, k][:, None]
        b[:, k + 1:] -= f * b[:, k][:, None]
    for k in range(n - 1, -1, -1):
        b[:, k] /= A[:, k, k]
        b[:, :k] -= A[:, :k, k] * b[:, k][:, None]
    return b


def condensed_rhs(prob, r_u, r_h):
    """g = sum_K P_K^T C_K A_K^-1 M_K r_K of an oracle problem (HDGProblem)."""
    p, R = prob.prm.p, reference_matrices(prob.prm.p)
    n, pp = R["n"], p + 1
    tau, g, H, ts = (LD(v) for v in (prob.prm.tau, prob.prm.g, prob.prm.H, prob.prm.tau_s))
    X, N = prob.X.astype(LD), prob.N
    f = prob.f_vertex[prob.md.cell_vertices].astype(LD)
    a, b, c, d = (X[:, 1, 0] - X[:, 0, 0], X[:, 2, 0] - X[:, 0, 0], X[:, 1, 1] - X[:, 0, 1], X[:, 2, 1] - X[:, 0, 1])
    det = a * d - b * c
    w = lambda v, M: v[:, None, None] * M  # noqa: E731
    M, Mf = w(det, R["M"]), sum(w(det * f[:, i], R["ML"][i]) for i in range(3))
    D = (w(d, R["Dxi"]) - w(c, R["Deta"]), w(a, R["Deta"]) - w(b, R["Dxi"]))
    u, v, h = slice(0, n), slice(n, 2 * n), slice(2 * n, 3 * n)
    A = np.zeros((N, 3 * n, 3 * n), LD)
    for s in (u, v, h):
        A[:, s, s] = M
    A[:, u, v], A[:, v, u] = -tau * Mf, tau * Mf
    C = np.zeros((N, 3 * pp, 3 * n), LD)
    for s, Ds in zip((u, v), D):
        A[:, s, h] = -tau * g * Ds.transpose(0, 2, 1)
        A[:, h, s] = tau * H * Ds
    for i in range(3):
        t, sl, Ni = X[:, (i + 2) % 3] - X[:, (i + 1) % 3], slice(i * pp, (i + 1) * pp), R["N"][i].T
        le = np.sqrt((t * t).sum(1))
        A[:, h, h] += tau * ts * w(le, R["E"][i])
        C[:, sl, u], C[:, sl, v], C[:, sl, h] = H * w(t[:, 1], Ni), -H * w(t[:, 0], Ni), ts * w(le, Ni)
    r = [(M * q[:, None].astype(LD)).sum(-1) for q in (r_u[:, 0], r_u[:, 1], r_h)]
    out = np.zeros(prob.n_trace, LD)
    np.add.at(out, prob.gdof, (C * solve(A, np.concatenate(r, 1))[:, None]).sum(-1))
    return out
