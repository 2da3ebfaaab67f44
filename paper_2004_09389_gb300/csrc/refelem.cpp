// Reference-element matrices of the library, by Gauss quadrature.
//
// Cell space P^p on the reference triangle (Eq. DG_space_def) with the
// equispaced Lagrange basis written in barycentric product form
//     phi_{ijk} = F_i(L0) F_j(L1) F_k(L2),   F_i(L) = prod_{s<i} (pL - s)/(s+1),
// with (i, j, k) = (p-a-b, a, b) for the node (a/p, b/p).  Trace space P^p on a
// facet (Eq. DG_trace_def) with the 1-D Lagrange basis at t_j = j/p.
// Triangle integrals use the collapsed Gauss-Legendre rule (xi = u,
// eta = v(1-u), weight (1-u)); edge integrals a Gauss-Legendre rule on [0, 1].
// Both are exact for the polynomial degrees involved (<= 2p+2).  Everything is formed in
// extended precision and rounded to FP64 once: the nodal matrices multiply the weak ones by
// M^-1, so that FP64 quadrature (a few 1e-16) left up to 4e-15 of relative error in the
// lifts, the same on every cell, and the recovered velocity two to six times as far off
// (242 cells, Courant 16: 3.7e-15 instead of 6e-16 at p = 1, 2.1e-14 instead of 1e-14 at p = 4).
// Extended precision is software on some hosts, so what follows from something else is not
// integrated: the reflection xi <-> eta maps the element onto itself, derivatives come from
// the nodes, and an edge sees its own p + 1 nodes (0.69 ms at p = 4 on Grace, 7.9 with every
// matrix integrated).
#include "common.h"

#include <cmath>
#include <limits>
#include <utility>

namespace hdg {

namespace {

using Real = long double;

// Gauss-Legendre nodes and weights on [0, 1] by Newton iteration on P_n (n >= 2).
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
        for (int it = 0; it < 8; ++it) {
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

// F_i and p dF_i/d(pL), i = 0..p, at pL = x
struct Factors {
    Real f[5], d[5];
    Factors(int p, Real x) {
        f[0] = 1.0L;
        d[0] = 0.0L;
        for (int s = 0; s < p; ++s) {
            const Real t = (x - s) / (s + 1);
            d[s + 1] = d[s] * t + f[s] * p / (s + 1);
            f[s + 1] = f[s] * t;
        }
    }
};

// the node that xi <-> eta maps node k to
int mirrored(int p, int k) {
    const int a = node_b(p, k), b = node_a(p, k);
    return b * (p + 1) - b * (b - 1) / 2 + a;
}

// The independent matrices in extended precision: M, ML_1, M1 and the nodal derivative Dx
struct Base {
    int p, n, pp;
    std::vector<Real> M, ML1, M1, Dx;
    explicit Base(int p_) : p(p_), n(n_cell_nodes(p_)), pp(p_ + 1) {
        M.assign(size_t(n) * n, 0.0L);
        ML1.assign(size_t(n) * n, 0.0L);
        M1.assign(size_t(pp) * pp, 0.0L);
        Dx.assign(size_t(n) * n, 0.0L);
        std::vector<Real> x, w, v(n), m(pp);
        gauss_legendre01(p + 2, x, w);
        for (size_t iu = 0; iu < x.size(); ++iu) {
            const Factors f1(p, p * x[iu]);
            for (size_t iv = 0; iv < x.size(); ++iv) {
                const Real eta = x[iv] * (1.0L - x[iu]), wt = w[iu] * w[iv] * (1.0L - x[iu]);
                const Factors f0(p, p * (1.0L - x[iu] - eta)), f2(p, p * eta);
                for (int k = 0; k < n; ++k) {
                    const int a = node_a(p, k), b = node_b(p, k);
                    v[k] = f0.f[p - a - b] * f1.f[a] * f2.f[b];
                }
                for (int i = 0; i < n; ++i) {
                    const Real wv = wt * v[i], wl = wv * x[iu];
                    for (int j = 0; j <= i; ++j) {
                        M[i * n + j] += wv * v[j];
                        ML1[i * n + j] += wl * v[j];
                    }
                }
            }
        }
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < i; ++j) {
                M[j * n + i] = M[i * n + j];
                ML1[j * n + i] = ML1[i * n + j];
            }
        for (size_t q = 0; q < x.size(); ++q) {
            for (int j = 0; j < pp; ++j) {
                m[j] = 1.0L;
                for (int k = 0; k <= p; ++k)
                    if (k != j) m[j] *= (p * x[q] - k) / (j - k);
            }
            for (int j = 0; j < pp; ++j)
                for (int k = 0; k < pp; ++k) M1[j * pp + k] += w[q] * m[j] * m[k];
        }
        // dL0/dxi = -1, dL1/dxi = 1; the entries that nodal_dx_nonzero leaves out vanish
        for (int i = 0; i < n; ++i) {
            const int ai = node_a(p, i), bi = node_b(p, i);
            const Factors f0(p, p - ai - bi), f1(p, ai), f2(p, bi);
            for (int j = 0; j < n; ++j) {
                const int a = node_a(p, j), b = node_b(p, j), c = p - a - b;
                Dx[i * n + j] = (f0.f[c] * f1.d[a] - f0.d[c] * f1.f[a]) * f2.f[b];
            }
        }
    }
    // A with rows and columns mirrored
    std::vector<Real> mirror(const std::vector<Real> &A) const {
        std::vector<Real> B(A.size());
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j) B[size_t(mirrored(p, i)) * n + mirrored(p, j)] = A[size_t(i) * n + j];
        return B;
    }
};

void rounded(const std::vector<Real> &a, std::vector<double> &b) { b.assign(a.begin(), a.end()); }

RefElem weak_matrices(const Base &q) {
    const int p = q.p, n = q.n, pp = q.pp;
    RefElem r;
    r.p = p;
    r.n = n;
    r.pp = pp;
    rounded(q.M, r.M);
    rounded(q.M1, r.M1);
    const std::vector<Real> ML2 = q.mirror(q.ML1);
    std::vector<Real> ML(size_t(3) * n * n), D(size_t(n) * n, 0.0L);
    for (int k = 0; k < n * n; ++k) {
        ML[k] = q.M[k] - q.ML1[k] - ML2[k];
        ML[n * n + k] = q.ML1[k];
        ML[2 * n * n + k] = ML2[k];
    }
    rounded(ML, r.ML);
    for (int k = 0; k < n; ++k)
        for (int j = 0; j < n; ++j)
            if (nodal_dx_nonzero(p, k, j))
                for (int i = 0; i < n; ++i) D[i * n + j] += q.M[i * n + k] * q.Dx[k * n + j];
    rounded(D, r.Dxi);
    rounded(q.mirror(D), r.Deta);
    r.E.assign(size_t(3) * n * n, 0.0);
    r.N.assign(size_t(3) * n * pp, 0.0);
    for (int i = 0; i < 3; ++i)
        for (int a = 0; a < pp; ++a)
            for (int j = 0; j < pp; ++j) {
                const int ka = edge_cell_node(p, i, a);
                r.N[(size_t(i) * n + ka) * pp + j] = r.M1[a * pp + j];
                r.E[(size_t(i) * n + ka) * n + edge_cell_node(p, i, j)] = r.M1[a * pp + j];
            }
    return r;
}

}  // namespace

RefElem build_ref_elem(int p) { return weak_matrices(Base(p)); }

NodalRef build_nodal_ref(int p, RefElem *weak) {
    const Base q(p);
    if (weak) *weak = weak_matrices(q);
    const int n = q.n, pp = q.pp;
    // [lift | ML1] = M^-1 [N_0 | N_1 | N_2 | ML_1]: Gauss-Jordan with partial pivoting
    const int w = 3 * pp + n;
    std::vector<Real> A(q.M), B(size_t(n) * w, 0.0L);
    for (int i = 0; i < 3; ++i)
        for (int a = 0; a < pp; ++a)
            for (int j = 0; j < pp; ++j) B[size_t(edge_cell_node(p, i, a)) * w + i * pp + j] = q.M1[a * pp + j];
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) B[size_t(i) * w + 3 * pp + j] = q.ML1[size_t(i) * n + j];
    for (int c = 0; c < n; ++c) {
        int piv = c;
        for (int i = c + 1; i < n; ++i)
            if (std::fabs(A[size_t(i) * n + c]) > std::fabs(A[size_t(piv) * n + c])) piv = i;
        for (int j = c; j < n; ++j) std::swap(A[size_t(c) * n + j], A[size_t(piv) * n + j]);
        for (int j = 0; j < w; ++j) std::swap(B[size_t(c) * w + j], B[size_t(piv) * w + j]);
        const Real d = 1.0L / A[size_t(c) * n + c];
        for (int j = c; j < n; ++j) A[size_t(c) * n + j] *= d;
        for (int j = 0; j < w; ++j) B[size_t(c) * w + j] *= d;
        for (int i = 0; i < n; ++i) {
            if (i == c) continue;
            const Real f = A[size_t(i) * n + c];
            for (int j = c; j < n; ++j) A[size_t(i) * n + j] -= f * A[size_t(c) * n + j];
            for (int j = 0; j < w; ++j) B[size_t(i) * w + j] -= f * B[size_t(c) * w + j];
        }
    }
    // Integration by parts on the reference element, edge normals times lengths (1, 1),
    // (-1, 0), (0, -1): Wx = -M^-1 Dxi^T = Dx - lift_0 + lift_1 on the edges' nodes
    std::vector<Real> ML1(size_t(n) * n), Wx(q.Dx);
    NodalRef r;
    r.lift.assign(size_t(3) * n * pp, 0.0);
    for (int i = 0; i < n; ++i) {
        for (int e = 0; e < 3; ++e)
            for (int j = 0; j < pp; ++j) {
                const Real l = B[size_t(i) * w + e * pp + j];
                r.lift[(size_t(e) * n + i) * pp + j] = double(l);
                if (e < 2) Wx[size_t(i) * n + edge_cell_node(p, e, j)] += e == 0 ? -l : l;
            }
        for (int j = 0; j < n; ++j) ML1[size_t(i) * n + j] = B[size_t(i) * w + 3 * pp + j];
    }
    rounded(q.Dx, r.Dx);
    rounded(q.mirror(q.Dx), r.Dy);
    rounded(ML1, r.ML1);
    rounded(q.mirror(ML1), r.ML2);
    rounded(Wx, r.Wx);
    rounded(q.mirror(Wx), r.Wy);
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
