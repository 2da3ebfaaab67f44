// Reference-element matrices of the library, by Gauss quadrature.
//
// Cell space P^p on the reference triangle (Eq. DG_space_def) with the
// equispaced Lagrange basis written in barycentric product form
//     phi_{ijk} = F_i(L0) F_j(L1) F_k(L2),   F_i(L) = prod_{s<i} (pL - s)/(s+1),
// with (i, j, k) = (p-a-b, a, b) for the node (a/p, b/p).  Trace space P^p on a
// facet (Eq. DG_trace_def) with the 1-D Lagrange basis at t_j = j/p.
// Triangle integrals use the collapsed Gauss-Legendre rule (xi = u,
// eta = v(1-u), weight (1-u)); edge integrals a Gauss-Legendre rule on [0, 1].
// Both are exact for the polynomial degrees involved (<= 2p+1).  Everything is formed in
// extended precision and rounded to FP64 once: the nodal matrices multiply the weak ones by
// M^-1, so that FP64 quadrature (a few 1e-16) left up to 4e-15 of relative error in the
// lifts, the same on every cell, and the recovered velocity two to six times as far off
// (242 cells, Courant 16: 3.7e-15 instead of 6e-16 at p = 1, 2.1e-14 instead of 1e-14 at p = 4).
#include "common.h"

#include <cmath>
#include <limits>
#include <utility>

namespace hdg {

namespace {

using Real = long double;

// Gauss-Legendre nodes and weights on [0, 1] by Newton iteration on P_n.
void gauss_legendre01(int n, std::vector<Real> &x, std::vector<Real> &w) {
    x.assign(n, 0.0L);
    w.assign(n, 0.0L);
    // P_n(z) and P_n'(z)
    auto legendre = [n](Real z, Real &p, Real &dp) {
        Real p0 = 1.0L;
        p = z;
        for (int k = 2; k <= n; ++k) {
            const Real p2 = ((2 * k - 1) * z * p - (k - 1) * p0) / k;
            p0 = p;
            p = p2;
        }
        dp = n * (z * p - p0) / (z * z - 1.0L);
    };
    for (int i = 0; i < n; ++i) {
        Real z = std::cos(3.14159265358979323846 * (i + 0.75) / (n + 0.5)), p, dp;
        for (int it = 0; it < 100; ++it) {
            legendre(z, p, dp);
            const Real dz = p / dp;
            z -= dz;
            if (std::fabs(dz) < 2 * std::numeric_limits<Real>::epsilon()) break;
        }
        legendre(z, p, dp);                            // the derivative at the converged node
        x[i] = 0.5L * (1.0L - z);
        w[i] = 1.0L / ((1.0L - z * z) * dp * dp);      // 2/((1-z^2)P'^2) on [-1,1], halved
    }
}

// F_i(L) and its derivative dF_i/dL
void factor(int p, int i, Real L, Real &f, Real &df) {
    f = 1.0L;
    df = 0.0L;
    for (int s = 0; s < i; ++s) {
        const Real t = (p * L - s) / (s + 1), dt = Real(p) / (s + 1);
        df = df * t + f * dt;
        f *= t;
    }
}

// basis values and xi/eta derivatives at (xi, eta)
void eval_basis(int p, Real xi, Real eta, std::vector<Real> &v, std::vector<Real> &dx, std::vector<Real> &dy) {
    int n = n_cell_nodes(p);
    v.resize(n); dx.resize(n); dy.resize(n);
    const Real L0 = 1.0L - xi - eta, L1 = xi, L2 = eta;
    int k = 0;
    for (int b = 0; b <= p; ++b) {
        for (int a = 0; a <= p - b; ++a, ++k) {
            int i0 = p - a - b, i1 = a, i2 = b;
            Real f0, d0, f1, d1, f2, d2;
            factor(p, i0, L0, f0, d0);
            factor(p, i1, L1, f1, d1);
            factor(p, i2, L2, f2, d2);
            v[k] = f0 * f1 * f2;
            dx[k] = -d0 * f1 * f2 + f0 * d1 * f2;   // dL0/dxi = -1, dL1/dxi = 1
            dy[k] = -d0 * f1 * f2 + f0 * f1 * d2;   // dL0/deta = -1, dL2/deta = 1
        }
    }
}

Real trace_basis(int p, int j, Real t) {
    Real v = 1.0L;
    for (int k = 0; k <= p; ++k)
        if (k != j) v *= (t - Real(k) / p) / (Real(j - k) / p);
    return v;
}

// the matrices of RefElem in extended precision
struct Weak {
    int n, pp;
    std::vector<Real> M, ML, Dxi, Deta, E, N, M1;
};
Weak weak_matrices(int p) {
    Weak r;
    r.n = n_cell_nodes(p);
    r.pp = p + 1;
    const int n = r.n, pp = r.pp;
    r.M.assign(n * n, 0.0L);
    r.ML.assign(3 * n * n, 0.0L);
    r.Dxi.assign(n * n, 0.0L);
    r.Deta.assign(n * n, 0.0L);
    r.E.assign(3 * n * n, 0.0L);
    r.N.assign(3 * n * pp, 0.0L);
    r.M1.assign(pp * pp, 0.0L);

    std::vector<Real> gx, gw;
    gauss_legendre01(p + 3, gx, gw);
    std::vector<Real> v, dx, dy;
    for (size_t iu = 0; iu < gx.size(); ++iu) {
        for (size_t iv = 0; iv < gx.size(); ++iv) {
            const Real xi = gx[iu], eta = gx[iv] * (1.0L - gx[iu]);
            const Real wt = gw[iu] * gw[iv] * (1.0L - gx[iu]);
            eval_basis(p, xi, eta, v, dx, dy);
            const Real L[3] = {1.0L - xi - eta, xi, eta};
            for (int a = 0; a < n; ++a) {
                for (int b = 0; b < n; ++b) {
                    const Real vv = wt * v[a] * v[b];
                    r.M[a * n + b] += vv;
                    for (int i = 0; i < 3; ++i) r.ML[(i * n + a) * n + b] += L[i] * vv;
                    r.Dxi[a * n + b] += wt * v[a] * dx[b];
                    r.Deta[a * n + b] += wt * v[a] * dy[b];
                }
            }
        }
    }
    std::vector<Real> ex, ew;
    gauss_legendre01(p + 2, ex, ew);
    const int V[3][2] = {{0, 0}, {1, 0}, {0, 1}};
    for (int i = 0; i < 3; ++i) {
        const int *A = V[(i + 1) % 3], *B = V[(i + 2) % 3];
        for (size_t q = 0; q < ex.size(); ++q) {
            const Real t = ex[q], wt = ew[q];
            eval_basis(p, A[0] + t * (B[0] - A[0]), A[1] + t * (B[1] - A[1]), v, dx, dy);
            for (int a = 0; a < n; ++a) {
                for (int b = 0; b < n; ++b) r.E[(i * n + a) * n + b] += wt * v[a] * v[b];
                for (int j = 0; j < pp; ++j) r.N[(i * n + a) * pp + j] += wt * v[a] * trace_basis(p, j, t);
            }
        }
    }
    for (size_t q = 0; q < ex.size(); ++q)
        for (int j = 0; j < pp; ++j)
            for (int k = 0; k < pp; ++k)
                r.M1[j * pp + k] += ew[q] * trace_basis(p, j, ex[q]) * trace_basis(p, k, ex[q]);
    return r;
}

}  // namespace

RefElem build_ref_elem(int p) {
    const Weak w = weak_matrices(p);
    RefElem r;
    r.p = p;
    r.n = w.n;
    r.pp = w.pp;
    auto round = [](const std::vector<Real> &a, std::vector<double> &b) { b.assign(a.begin(), a.end()); };
    round(w.M, r.M);
    round(w.ML, r.ML);
    round(w.Dxi, r.Dxi);
    round(w.Deta, r.Deta);
    round(w.E, r.E);
    round(w.N, r.N);
    round(w.M1, r.M1);
    return r;
}

NodalRef build_nodal_ref(int p) {
    const Weak re = weak_matrices(p);
    const int n = re.n, pp = re.pp;
    NodalRef r;
    r.Dx.assign(size_t(n) * n, 0.0);
    r.Dy.assign(size_t(n) * n, 0.0);
    std::vector<Real> v, dx, dy;
    int k = 0;
    for (int b = 0; b <= p; ++b)
        for (int a = 0; a <= p - b; ++a, ++k) {
            eval_basis(p, Real(a) / p, Real(b) / p, v, dx, dy);
            for (int j = 0; j < n; ++j) {
                // the entries that nodal_dx_nonzero / nodal_dy_nonzero leave out vanish identically
                r.Dx[size_t(k) * n + j] = double(dx[j]);
                r.Dy[size_t(k) * n + j] = double(dy[j]);
            }
        }
    // [lift | ML1 | ML2 | -Wx | -Wy] = M^-1 [N_0 | N_1 | N_2 | ML_1 | ML_2 | Dxi^T | Deta^T]: Gauss-Jordan with
    // partial pivoting in extended precision, rounded once
    const int w = 3 * pp + 4 * n;
    std::vector<Real> A(size_t(n) * n), B(size_t(n) * w);
    for (int i = 0; i < n; ++i) {
        for (int j = 0; j < n; ++j) A[size_t(i) * n + j] = re.M[size_t(i) * n + j];
        for (int e = 0; e < 3; ++e)
            for (int j = 0; j < pp; ++j)
                B[size_t(i) * w + e * pp + j] = re.N[(size_t(e) * n + i) * pp + j];
        for (int l = 0; l < 2; ++l)
            for (int j = 0; j < n; ++j)
                B[size_t(i) * w + 3 * pp + l * n + j] = re.ML[(size_t(l + 1) * n + i) * n + j];
        for (int j = 0; j < n; ++j) {
            B[size_t(i) * w + 3 * pp + 2 * n + j] = re.Dxi[size_t(j) * n + i];
            B[size_t(i) * w + 3 * pp + 3 * n + j] = re.Deta[size_t(j) * n + i];
        }
    }
    for (int c = 0; c < n; ++c) {
        int piv = c;
        for (int i = c + 1; i < n; ++i)
            if (std::fabs(A[size_t(i) * n + c]) > std::fabs(A[size_t(piv) * n + c])) piv = i;
        for (int j = 0; j < n; ++j) std::swap(A[size_t(c) * n + j], A[size_t(piv) * n + j]);
        for (int j = 0; j < w; ++j) std::swap(B[size_t(c) * w + j], B[size_t(piv) * w + j]);
        const Real d = 1.0L / A[size_t(c) * n + c];
        for (int j = 0; j < n; ++j) A[size_t(c) * n + j] *= d;
        for (int j = 0; j < w; ++j) B[size_t(c) * w + j] *= d;
        for (int i = 0; i < n; ++i) {
            if (i == c) continue;
            const Real f = A[size_t(i) * n + c];
            for (int j = 0; j < n; ++j) A[size_t(i) * n + j] -= f * A[size_t(c) * n + j];
            for (int j = 0; j < w; ++j) B[size_t(i) * w + j] -= f * B[size_t(c) * w + j];
        }
    }
    r.lift.assign(size_t(3) * n * pp, 0.0);
    r.ML1.assign(size_t(n) * n, 0.0);
    r.ML2.assign(size_t(n) * n, 0.0);
    r.Wx.assign(size_t(n) * n, 0.0);
    r.Wy.assign(size_t(n) * n, 0.0);
    for (int i = 0; i < n; ++i) {
        for (int e = 0; e < 3; ++e)
            for (int j = 0; j < pp; ++j) r.lift[(size_t(e) * n + i) * pp + j] = double(B[size_t(i) * w + e * pp + j]);
        for (int j = 0; j < n; ++j) {
            r.ML1[size_t(i) * n + j] = double(B[size_t(i) * w + 3 * pp + j]);
            r.ML2[size_t(i) * n + j] = double(B[size_t(i) * w + 3 * pp + n + j]);
            r.Wx[size_t(i) * n + j] = -double(B[size_t(i) * w + 3 * pp + 2 * n + j]);
            r.Wy[size_t(i) * n + j] = -double(B[size_t(i) * w + 3 * pp + 3 * n + j]);
        }
    }
    return r;
}

std::vector<double> NodalRef::packed() const {
    std::vector<double> out;
    for (const std::vector<double> *m : {&Dx, &Dy, &lift, &ML1, &ML2, &Wx, &Wy}) out.insert(out.end(), m->begin(), m->end());
    return out;
}

std::vector<double> RefElem::packed() const {
    std::vector<double> out;
    out.insert(out.end(), M.begin(), M.end());
    out.insert(out.end(), ML.begin(), ML.end());
    out.insert(out.end(), Dxi.begin(), Dxi.end());
    out.insert(out.end(), Deta.begin(), Deta.end());
    out.insert(out.end(), E.begin(), E.end());
    out.insert(out.end(), N.begin(), N.end());
    out.insert(out.end(), M1.begin(), M1.end());
    return out;
}

}  // namespace hdg
