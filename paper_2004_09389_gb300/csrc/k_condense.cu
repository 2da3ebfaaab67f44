// Static condensation (Sec. 4.2) and assembly of the facet-row trace operator.
//
// Per cell K, with u_perp = (-u_y, u_x), the cell rows of the upwind HDG form
// (Eq. bilinear_HDG_upwind, ABCM split of Eq. ABCMform / App. B, Coriolis implicit)
// in the integrated-by-parts form
//   momentum: (u,w) + tau (f u_perp, w) - tau g (h, div w)         + tau g <lambda, w.n>
//   mass:     (h,psi) + tau H (div u, psi) + tau tau_s <h, psi>_dK - tau tau_s <lambda, psi>
//   facet:    <H u.n + tau_s h, mu> - tau_s <lambda, mu>
// i.e. A_K q + B_K lambda = Mass_K r on the cell and C_K q - Mt_K lambda on its
// facets, are condensed to X_B = A^-1 B, R_M = A^-1 Mass and
//   S_K = Mt_K + C_K X_B      (the cell's part of Eq. schur_system)
//   W_K = C_K R_M             (step 1: g = sum_K P_K^T W_K r_K)
// R_M and X_B serve step 3 (Eq. reconstruct_solution): q = R_M r - X_B lambda_K.
// The velocity is eliminated first, in function space, in FP64 (condense_nodal_kernel).
// The two-float handles keep S_K, X_B and, instead of R_M and W_K, what their cell solve
// takes: the h rows of R_M and the inverse of the velocity block (P and Q).
#include "common.h"

namespace hdg {

namespace {

template <int P>
struct Sz {
    static constexpr int PP = P + 1;
    static constexpr int NP = (P + 1) * (P + 2) / 2;
    static constexpr int NK = 3 * NP;
    static constexpr int M = 3 * PP;
};

// ---------------------------------------------------------------- condensation in function space
// Every cell matrix multiplied by M_K^-1, so that the cell equations act on
// nodal values and the reference matrices are the same for every cell:
//   u + tau F u_perp + tau g G h = r_u - b_u,   h + tau H div u + tau tau_s E h = r_h - b_h
// with F the projected multiplication by f, G the weak gradient, E the lifted edge
// traces and (b_u, b_h) = B^ lambda.  With R = (I + tau F J)^-1 = [P Q; -Q P],
// P = (I + tau^2 F^2)^-1, Q = tau F P, the velocity is eliminated first,
//   T = tau g R G,   S = I + tau tau_s E - tau H div T,   h = S^-1 (r_h - tau H div R r_u),
//   u = R r_u - T h,
// so that a cell takes two inverses of n_p x n_p instead of one of 3 n_p x 3 n_p.
// Where f is constant on every cell (FC; decided at set-up), F = f and P, Q are
// numbers: one inverse.  X_B = A^-1 B, R_M = A^-1 Mass and S_K = Mt_K + C X_B follow
// column by column, W_K = C R_M row by row.
//
// One thread per column of a cell, kCondCells<P> cells per block with the cell as
// the fastest thread index (shared-memory reads without bank conflicts, global
// writes in runs of neighbouring cells).  The FP64 pipe is the bound (1.05 TFLOP/s
// measured, one warp instruction in about 77 cycles per scheduler), so the split is
// the one that keeps the warps full (at p = 3 8 x 10 columns up to S, 8 x 12 for X_B
// and all 8 x 30 of R_M dealt to the 96 threads) and what need not be FP64 is not: the
// conversions to float pairs, the correction of the refinement, pivot tests.  The h
// columns of R_M are S^-1 as it stands, and R_M's h rows are not refined (step 1 and
// the recovery of the two-float handles are as exact either way, and so is the FP64
// recovery).  20,480 cells at p = 3, two-float, f varying: 1,345 us instead of 1,773 (one pass
// of 10 of 12 columns per component of R_M, all of them refined in FP64, a full division
// per pivot and column, two products where column k meets the pivot's).  FP64, 32,768 cells at
// p = 2, 3, 4: 518, 1,561 and 4,194 us (f varying 700, 2,324, 6,458), with W_K from the columns of
// R_M 559, 1,708 and 4,752 (712, 2,385, 6,763), by elimination of the whole augmented cell
// system [A | B | Mass], one cell per block, 2,587, 6,629 and 16,949.
template <int P> constexpr int kCondCells = P == 1 ? 16 : P == 2 ? 10 : P == 3 ? 8 : 6;
constexpr int kCondThreads = 96;

struct NodalArgs {
    int N;
    double tau, g, H, ts;
    const double *nref;     // packed nodal reference matrices
    const double *M1;       // [PP][PP] edge mass matrix
    const double *X;        // [N][3][2]
    const double *fcell;    // [N][3]
    double *Xb, *W, *Scell;            // FP64 handles (Scell: both)
    double *Rh, *Ru, *PQ;              // FP64 handles: the h rows of R_M, its velocity rows (or null) or
                                       // else (f varying over a cell) Q, P - Q, P + Q
    float2 *Xb2, *Hr2, *lgeo;          // two-float handles: X_B, the h rows of R_M, the cell
    float4 *PQ2;                       // weights and (f varying over a cell) P, Q
    int32_t *status;
};

// 1 / d by Newton's iteration from a single-precision reciprocal: two steps from 2^-23
// (four FMAs; the division takes about twice as many FP64 instructions)
__device__ __forceinline__ double reciprocal(double d) {
    const unsigned ex = (unsigned(__double2hiint(d)) >> 20) & 0x7ffu;
    if (ex - 923u > 200u) return 1.0 / d;                      // outside 2^-100 .. 2^100
    double r = join(make_float2(__frcp_rn(to_float(d)), 0.0f));
    r = fma(r, fma(-d, r, 1.0), r);
    return fma(r, fma(-d, r, 1.0), r);
}

// In-place inverse of the n x n matrices A[(i * n + j) * CC + c] of the block's cells
// by Gauss-Jordan elimination with partial pivoting; thread (c, j) owns column j.
// Every thread of the block calls it (on: the thread owns a column); piv is shared
// scratch [n][CC].  Sets bad on a zero pivot.
template <int n, int CC>
__device__ __forceinline__ void block_inverse(double *A, int c, int j, bool on, int *piv, int *bad) {
    for (int k = 0; k < n; ++k) {
        __syncthreads();
        double f[n];
        int p = k;
        if (on) {
            // the pivot row by magnitude (the high words order like the values)
            int best = -1;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                f[i] = A[(i * n + k) * CC + c];
                const int m = __double2hiint(f[i]) & 0x7fffffff;
                if (i >= k && m > best) {
                    best = m;
                    p = i;
                }
            }
        }
        __syncthreads();                       // column k has been read
        if (on) {
            double d = 0.0, fk = 0.0;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                if (i == p) d = f[i];
                if (i == k) fk = f[i];
            }
            // (the exponent first: comparisons take the FP64 pipe)
            const unsigned ex = (unsigned(__double2hiint(d)) >> 20) & 0x7ffu;
            if (ex - 27u > 2019u && !(fabs(d) > 1e-300)) *bad = 1;
            const double r = reciprocal(d);
            double *a = A + j * CC + c;
            const double akj = a[k * n * CC], apj = a[p * n * CC];
            if (p != k) a[p * n * CC] = akj;   // the rows swapped
            const double row = j == k ? r : apj * r;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const double fi = i == p ? fk : f[i];   // column k after the swap
                const double aij = a[i * n * CC];
                a[i * n * CC] = i == k ? row : fma(-fi, row, j == k ? 0.0 : aij);   // (j == k: row = r)
            }
            if (j == 0) piv[k * CC + c] = p;
        }
    }
    __syncthreads();
    // the row swaps, undone on the columns in reverse order: column j goes to place q
    double col[n];
    int q = j;
    if (on) {
        for (int k = n - 1; k >= 0; --k) {
            const int p = piv[k * CC + c];
            q = q == k ? p : q == p ? k : q;
        }
#pragma unroll
        for (int i = 0; i < n; ++i) col[i] = A[(i * n + j) * CC + c];
    }
    __syncthreads();
    if (on) {
#pragma unroll
        for (int i = 0; i < n; ++i) A[(i * n + q) * CC + c] = col[i];
    }
    __syncthreads();
}

// Keeps the compiler from moving shared-memory loads of later rows above this point
// (at p = 4 it would otherwise hold whole matrices in registers and spill).
__device__ __forceinline__ void row_fence() { asm volatile("" ::: "memory"); }

// rh += div of the contravariant velocity of (wx, wy) scaled by the weights g00 .. g11
// (nodal derivatives, the entries that vanish left out)
template <int P>
__device__ __forceinline__ void add_div(const double *ref, double g00, double g01, double g10, double g11,
                                        const double (&wx)[Sz<P>::NP], const double (&wy)[Sz<P>::NP],
                                        double (&rh)[Sz<P>::NP]) {
    constexpr int NP = Sz<P>::NP;
    constexpr NodalOffsets O = nodal_offsets(P);
    double c1[NP], c2[NP];
#pragma unroll
    for (int b = 0; b < NP; ++b) {
        c1[b] = fma(g00, wx[b], g10 * wy[b]);
        c2[b] = fma(g01, wx[b], g11 * wy[b]);
    }
    static_for<NP>([&](auto ia_) {
        constexpr int ia = decltype(ia_)::value;
        row_fence();
        static_for<NP>([&](auto ib_) {
            constexpr int ib = decltype(ib_)::value;
            if constexpr (nodal_dx_nonzero(P, ia, ib)) rh[ia] = fma(ref[O.Dx + ia * NP + ib], c1[ib], rh[ia]);
            if constexpr (nodal_dy_nonzero(P, ia, ib)) rh[ia] = fma(ref[O.Dy + ia * NP + ib], c2[ib], rh[ia]);
        });
    });
}

// h = S^-1 rh for cell c of the block's matrices, the explicit inverse
template <int NP, int CC>
__device__ __forceinline__ void inverse_product(const double *Ss, int c, const double (&rh)[NP], double (&h)[NP]) {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        row_fence();
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < NP; ++k) v = fma(Ss[(i * NP + k) * CC + c], rh[k], v);
        h[i] = v;
    }
}

// One step of iterative refinement of h = S^-1 rh: the residual in FP64 from S itself (So)
// and its correction, 1e-14 of h, with the inverse rounded to FP32 (Sf).  The explicit inverse
// alone leaves S_K about 20 times less exact than an elimination of the whole cell system
// (p = 3, Courant 16: S_K applied to a nearly constant trace off by 1e-12 instead of
// 7e-14; one step brings it to 2e-14).
template <int NP, int CC>
__device__ __forceinline__ void refine(const double *So, const float *Sf, int c, const double (&rh)[NP],
                                       double (&h)[NP]) {
    float res[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        row_fence();
        double v = rh[i];
#pragma unroll
        for (int k = 0; k < NP; ++k) v = fma(-So[(i * NP + k) * CC + c], h[k], v);
        res[i] = to_float(v);
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        row_fence();
        float v = 0.0f;
#pragma unroll
        for (int k = 0; k < NP; ++k) v = fmaf(Sf[(i * NP + k) * CC + c], res[k], v);
        h[i] += join(make_float2(v, 0.0f));
    }
}

// (wx, wy) -= T h
template <int NP, int CC>
__device__ __forceinline__ void subtract_gradient(const double *Ts, int c, const double (&h)[NP], double (&wx)[NP],
                                                  double (&wy)[NP]) {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        row_fence();
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            wx[i] = fma(-Ts[(i * NP + k) * CC + c], h[k], wx[i]);
            wy[i] = fma(-Ts[((NP + i) * NP + k) * CC + c], h[k], wy[i]);
        }
    }
}

// edge weights of C: (H t_y, -H t_x, tau_s |e|) of edge e of cell K
__device__ __forceinline__ void edge_weights(const NodalArgs &a, const double *geo, int CC, int c, int K, int e,
                                             double (&w)[3]) {
    const double *x = a.X + size_t(K) * 6;
    const double det = (x[2] - x[0]) * (x[5] - x[1]) - (x[4] - x[0]) * (x[3] - x[1]);
    w[0] = a.H * det * geo[(4 + 3 * e) * CC + c];
    w[1] = a.H * det * geo[(5 + 3 * e) * CC + c];
    w[2] = a.ts * det * geo[(6 + 3 * e) * CC + c];
}

// row (edge e, node jj) of C q into out[row * ld]; diag is added to the rows of edge e0
// (diag times column jj0 of the edge mass matrix)
template <int P>
__device__ __forceinline__ void c_rows(const double *m1, const double (&wn)[3][3], const double (&qx)[Sz<P>::NP],
                                       const double (&qy)[Sz<P>::NP], const double (&qh)[Sz<P>::NP], int e0, int jj0,
                                       double diag, double *out, size_t ld) {
    constexpr int PP = P + 1;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        row_fence();
        double fl[PP];
#pragma unroll
        for (int jb = 0; jb < PP; ++jb) {
            const int b = edge_cell_node(P, e, jb);
            fl[jb] = fma(wn[e][0], qx[b], fma(wn[e][1], qy[b], wn[e][2] * qh[b]));
        }
#pragma unroll
        for (int jj = 0; jj < PP; ++jj) {
            double v = e == e0 ? diag * m1[jj * PP + jj0] : 0.0;
#pragma unroll
            for (int jb = 0; jb < PP; ++jb) v = fma(m1[jb * PP + jj], fl[jb], v);
            out[size_t(e * PP + jj) * ld] = v;
        }
    }
}

// Row (edge e, node jj) of W_K = C R_M for cell c of the block's matrices: C's row with the
// velocity eliminated, k = C_h - C_u T, times S^-1 with one refinement step (as in refine, from
// the left), gives the entries w for r_h; (C_u - w tau H div) R is those for r_u, formed here where
// R is two numbers (FC), else column by column from w (w_column).  By rows
// every entry is exact to its own rounding: from the columns of R_M, each refined, the
// condensed right-hand side of smooth r_h alone was up to 20 times as far off (p = 4, Courant
// 16: 6.8e-15), and unrefined that of smooth r_u and r_h 1.1e-13.
template <int P, bool FC, int CC>
__device__ __forceinline__ void w_row(const double *ref, const double *m1, const double *Ss, const double *So,
                                      const float *Sf, const double *Ts, int c, int e, int jj, double w0, double w1,
                                      double w2, double g00, double g01, double g10, double g11, double kap, double fk,
                                      double *out, size_t ld, double (&w)[Sz<P>::NP]) {
    constexpr int PP = P + 1, NP = Sz<P>::NP;
    constexpr NodalOffsets O = nodal_offsets(P);
    auto mu = [&](int i) {                     // the edge mass matrix's column jj at cell node i
        const int pos = e == 0 ? node_edge_pos(P, 0, i) : e == 1 ? node_edge_pos(P, 1, i) : node_edge_pos(P, 2, i);
        return pos >= 0 ? m1[pos * PP + jj] : 0.0;
    };
    double k[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        k[i] = w2 * mu(i);
        w[i] = 0.0;
    }
#pragma unroll
    for (int jb = 0; jb < PP; ++jb) {
        row_fence();
        const int b = edge_cell_node(P, e, jb);
        const double x = w0 * m1[jb * PP + jj], y = w1 * m1[jb * PP + jj];
#pragma unroll
        for (int j = 0; j < NP; ++j)
            k[j] = fma(-x, Ts[(b * NP + j) * CC + c], fma(-y, Ts[((NP + b) * NP + j) * CC + c], k[j]));
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        row_fence();
#pragma unroll
        for (int j = 0; j < NP; ++j) w[j] = fma(k[i], Ss[(i * NP + j) * CC + c], w[j]);
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        row_fence();
#pragma unroll
        for (int j = 0; j < NP; ++j) k[j] = fma(-w[i], So[(i * NP + j) * CC + c], k[j]);
    }
    float r[NP], d[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        r[i] = to_float(k[i]);
        d[i] = 0.0f;
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        row_fence();
#pragma unroll
        for (int j = 0; j < NP; ++j) d[j] = fmaf(r[i], Sf[(i * NP + j) * CC + c], d[j]);
    }
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        w[j] += join(make_float2(d[j], 0.0f));
        out[size_t(2 * NP + j) * ld] = w[j];
    }
    if constexpr (FC) {
        double vx[NP], vy[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) vx[j] = vy[j] = 0.0;
        static_for<NP>([&](auto ia_) {
            constexpr int ia = decltype(ia_)::value;
            row_fence();
            static_for<NP>([&](auto ib_) {
                constexpr int ib = decltype(ib_)::value;
                if constexpr (nodal_dx_nonzero(P, ia, ib)) vx[ib] = fma(ref[O.Dx + ia * NP + ib], w[ia], vx[ib]);
                if constexpr (nodal_dy_nonzero(P, ia, ib)) vy[ib] = fma(ref[O.Dy + ia * NP + ib], w[ia], vy[ib]);
            });
        });
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            const double q = mu(j), x = fma(w0, q, fma(g00, vx[j], g01 * vy[j])), y = fma(w1, q, fma(g10, vx[j], g11 * vy[j]));
            out[size_t(j) * ld] = fma(kap, x, -fk * y);
            out[size_t(NP + j) * ld] = fma(fk, x, kap * y);
        }
    }
}

// Column of W_K for a unit vector in r_u: C_u (wx, wy) + w rh with (wx, wy) its velocity R e and rh =
// -tau H div R e, the rows w of the cell from shared memory ([M][NP][CC])
template <int P, int CC>
__device__ __forceinline__ void w_column(const double *m1, const double *ws, int c, const double (&wn)[3][3],
                                         const double (&wx)[Sz<P>::NP], const double (&wy)[Sz<P>::NP],
                                         const double (&rh)[Sz<P>::NP], double *out, size_t ld) {
    constexpr int PP = P + 1, NP = Sz<P>::NP;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        row_fence();
        double fl[PP];
#pragma unroll
        for (int jb = 0; jb < PP; ++jb) {
            const int b = edge_cell_node(P, e, jb);
            fl[jb] = fma(wn[e][0], wx[b], wn[e][1] * wy[b]);
        }
#pragma unroll
        for (int jj = 0; jj < PP; ++jj) {
            double v = 0.0;
#pragma unroll
            for (int jb = 0; jb < PP; ++jb) v = fma(m1[jb * PP + jj], fl[jb], v);
#pragma unroll
            for (int i = 0; i < NP; ++i) v = fma(ws[((e * PP + jj) * NP + i) * CC + c], rh[i], v);
            out[size_t(e * PP + jj) * ld] = v;
        }
    }
}

// shared memory of the kernel below, in doubles
template <int P, bool FC>
struct CondSmem {
    static constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2, NN = NP * NP, CC = kCondCells<P>;
    static constexpr int oRef = 0, oM1 = nodal_offsets(P).total, oGeo = oM1 + PP * PP;
    static constexpr int nGeo = 4 + 9 + 2 + 3;                     // j, edge weights, R (FC), f
    static constexpr int oS = oGeo + nGeo * CC, oT = oS + NN * CC, oSo = oT + 2 * NN * CC;
    static constexpr int oSf = oSo + NN * CC, nSf = (NN * CC + 1) / 2;                     // (oSf: floats)
    // the rows w of W_K take the place of So and Sf (which they outgrow at p = 1)
    static constexpr int nW = FC ? 0 : 3 * PP * NP * CC, oP = oSo + (nW > NN * CC + nSf ? nW : NN * CC + nSf);
    static constexpr int oQ = oP + (FC ? 0 : NN * CC), total = oQ + (FC ? 0 : NN * CC);
};

// blocks per SM that the kernel is compiled for (as many as the shared memory admits from p = 3
// on; 0: the compiler's choice, which suits the two-float instances but the one at p = 3 with f
// varying: 1,377 instead of 1,398 us on 20,480 cells, by how the last of its blocks fall)
template <int P, bool FC, bool FF>
constexpr int kCondPerSM = FF ? (P == 3 && !FC ? 4 : 0) : P == 1 ? 10 : P == 2 ? 7 : P == 3 ? (FC ? 5 : 4) : (FC ? 3 : 2);

template <int P, bool FC, bool FF>
__global__ void __launch_bounds__(kCondThreads, kCondPerSM<P, FC, FF>) condense_nodal_kernel(NodalArgs a) {
    using L = CondSmem<P, FC>;
    constexpr int PP = P + 1, NP = L::NP, NK = 3 * NP, M = 3 * PP, CC = L::CC;
    constexpr NodalOffsets O = nodal_offsets(P);
    extern __shared__ double sm[];
    double *ref = sm + L::oRef, *m1 = sm + L::oM1, *geo = sm + L::oGeo;
    double *Ss = sm + L::oS, *Ts = sm + L::oT, *So = sm + L::oSo, *Ps = sm + L::oP, *Qs = sm + L::oQ;
    float *Sf = reinterpret_cast<float *>(sm + L::oSf);
    __shared__ int piv[NP * CC];
    __shared__ int bad;
    const int t = threadIdx.x, c = t % CC, j = t / CC;
    const int K = blockIdx.x * CC + c;
    const bool cell = K < a.N, on = cell && j < NP;
    if (t == 0) bad = 0;
    for (int k = t; k < O.total; k += kCondThreads) ref[k] = a.nref[k];
    for (int k = t; k < PP * PP; k += kCondThreads) m1[k] = a.M1[k];
    // geometry of the cell, [entry][CC]: J^-T (0..3), per edge 1/det times (t_y, -t_x, |e|)
    // (4..12), P and Q where f is constant on the cell (13, 14), tau times f_0, f_1 - f_0,
    // f_2 - f_0 (15..17)
    if (cell && j == 0) {
        const double *x = a.X + size_t(K) * 6;
        const double J00 = x[2] - x[0], J01 = x[4] - x[0], J10 = x[3] - x[1], J11 = x[5] - x[1];
        const double s = 1.0 / (J00 * J11 - J01 * J10);
        geo[0 * CC + c] = J11 * s;
        geo[1 * CC + c] = -J10 * s;
        geo[2 * CC + c] = -J01 * s;
        geo[3 * CC + c] = J00 * s;
        for (int i = 0; i < 3; ++i) {
            const int v1 = (i + 1) % 3, v2 = (i + 2) % 3;
            const double tx = x[2 * v2] - x[2 * v1], ty = x[2 * v2 + 1] - x[2 * v1 + 1];
            geo[(4 + 3 * i) * CC + c] = s * ty;
            geo[(5 + 3 * i) * CC + c] = -s * tx;
            geo[(6 + 3 * i) * CC + c] = s * sqrt(tx * tx + ty * ty);
        }
        const double f0 = a.fcell[size_t(K) * 3];
        const double f = a.tau * f0, kap = 1.0 / fma(f, f, 1.0);
        geo[13 * CC + c] = kap;
        geo[14 * CC + c] = f * kap;
        geo[15 * CC + c] = f;
        geo[16 * CC + c] = a.tau * (a.fcell[size_t(K) * 3 + 1] - f0);
        geo[17 * CC + c] = a.tau * (a.fcell[size_t(K) * 3 + 2] - f0);
    }
    __syncthreads();
    const double tg = a.tau * a.g, tH = a.tau * a.H;
    const double j00 = geo[0 * CC + c], j01 = geo[1 * CC + c], j10 = geo[2 * CC + c], j11 = geo[3 * CC + c];

    // ---- R: P and Q (f varying over the cell); tau F waits in T's place
    if constexpr (!FC) {
        double col[NP];
        if (on) {
            const double f0 = geo[15 * CC + c], f1 = geo[16 * CC + c], f2 = geo[17 * CC + c];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                col[i] = fma(f1, ref[O.ML1 + i * NP + j], f2 * ref[O.ML2 + i * NP + j]);
                if (i == j) col[i] += f0;
                Ts[(i * NP + j) * CC + c] = col[i];
            }
        }
        __syncthreads();
        if (on) {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                row_fence();
                double v = i == j ? 1.0 : 0.0;
#pragma unroll
                for (int k = 0; k < NP; ++k) v = fma(Ts[(i * NP + k) * CC + c], col[k], v);
                Ps[(i * NP + j) * CC + c] = v;
            }
        }
        block_inverse<NP, CC>(Ps, c, j, on, piv, &bad);
        if (on) {
#pragma unroll
            for (int i = 0; i < NP; ++i) col[i] = Ps[(i * NP + j) * CC + c];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                row_fence();
                double v = 0.0;
#pragma unroll
                for (int k = 0; k < NP; ++k) v = fma(Ts[(i * NP + k) * CC + c], col[k], v);
                Qs[(i * NP + j) * CC + c] = v;
            }
        }
        __syncthreads();
    }
    const double kap = geo[13 * CC + c], fk = geo[14 * CC + c];

    // ---- T = tau g R G and S, column j
    if (on) {
        double tx[NP], ty[NP], s[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) tx[i] = ty[i] = 0.0;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            row_fence();
            const double wx = ref[O.Wx + k * NP + j], wy = ref[O.Wy + k * NP + j];
            const double gx = tg * fma(j00, wx, j01 * wy), gy = tg * fma(j10, wx, j11 * wy);
            if constexpr (FC) {
                tx[k] = fma(kap, gx, fk * gy);
                ty[k] = fma(kap, gy, -fk * gx);
            } else {
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    const double p = Ps[(i * NP + k) * CC + c], q = Qs[(i * NP + k) * CC + c];
                    tx[i] = fma(p, gx, fma(q, gy, tx[i]));
                    ty[i] = fma(p, gy, fma(-q, gx, ty[i]));
                }
            }
        }
        const double tts = a.tau * a.ts;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            s[i] = i == j ? 1.0 : 0.0;
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const int pos = node_edge_pos(P, e, j);
                if (pos >= 0) s[i] = fma(tts * geo[(6 + 3 * e) * CC + c], ref[O.lift + (e * NP + i) * PP + pos], s[i]);
            }
        }
        add_div<P>(ref, -tH * j00, -tH * j01, -tH * j10, -tH * j11, tx, ty, s);
        // (T overwrites tau F, whose last readers are behind the barrier above)
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            Ts[(i * NP + j) * CC + c] = tx[i];
            Ts[((NP + i) * NP + j) * CC + c] = ty[i];
            Ss[(i * NP + j) * CC + c] = s[i];
            So[(i * NP + j) * CC + c] = s[i];
        }
    }
    block_inverse<NP, CC>(Ss, c, j, on, piv, &bad);
    if (bad) {
        if (t == 0) atomicOr(a.status, 1);
        return;
    }
    if (on) {
#pragma unroll
        for (int i = 0; i < NP; ++i) Sf[(i * NP + j) * CC + c] = to_float(Ss[(i * NP + j) * CC + c]);
    }
    __syncthreads();

    double wn[3][3];
#pragma unroll
    for (int e = 0; e < 3; ++e) edge_weights(a, geo, CC, c, cell ? K : 0, e, wn[e]);
    const size_t N = a.N;
    // ---- X_B and S_K, column (edge e, trace node jj)
    if (cell && j < M) {
        const int e = j / PP, jj = j % PP;
        const double bx = tg * geo[(4 + 3 * e) * CC + c], by = tg * geo[(5 + 3 * e) * CC + c];
        const double bh = -a.tau * a.ts * geo[(6 + 3 * e) * CC + c];
        double wx[NP], wy[NP], rh[NP], h[NP];
        if constexpr (FC) {
            const double rx = fma(kap, bx, fk * by), ry = fma(kap, by, -fk * bx);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const double l = ref[O.lift + (e * NP + i) * PP + jj];
                wx[i] = rx * l;
                wy[i] = ry * l;
                rh[i] = bh * l;
            }
        } else {
            double pl[NP], ql[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) pl[i] = ql[i] = 0.0;
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                row_fence();
                const double l = ref[O.lift + (e * NP + k) * PP + jj];
                rh[k] = bh * l;
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    pl[i] = fma(Ps[(i * NP + k) * CC + c], l, pl[i]);
                    ql[i] = fma(Qs[(i * NP + k) * CC + c], l, ql[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                wx[i] = fma(bx, pl[i], by * ql[i]);
                wy[i] = fma(by, pl[i], -bx * ql[i]);
            }
        }
        add_div<P>(ref, -tH * j00, -tH * j01, -tH * j10, -tH * j11, wx, wy, rh);
        inverse_product<NP, CC>(Ss, c, rh, h);
        refine<NP, CC>(So, Sf, c, rh, h);
        subtract_gradient<NP, CC>(Ts, c, h, wx, wy);
        if constexpr (FF) {
            constexpr int CPb = (M + 1) / 2;
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const double v[3] = {wx[i], wy[i], h[i]};
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    a.Xb2[2 * ff_pair_index(size_t(K), size_t(q * NP + i) * CPb + j / 2, size_t(NK) * CPb) + j % 2] =
                        split(v[q]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                a.Xb[(size_t(i) * M + j) * N + K] = wx[i];
                a.Xb[(size_t(NP + i) * M + j) * N + K] = wy[i];
                a.Xb[(size_t(2 * NP + i) * M + j) * N + K] = h[i];
            }
        }
        c_rows<P>(m1, wn, wx, wy, h, e, jj, e == 0 ? wn[0][2] : e == 1 ? wn[1][2] : wn[2][2], a.Scell + size_t(K) * M * M + j, M);
    }
    if constexpr (!FF) {
        // ---- W_K, row (edge e, trace node jj)
        double wr[NP];
        if (cell && j < M) {
            const int e = j / PP, jj = j % PP;
            auto of_edge = [&](int q) { return e == 0 ? wn[0][q] : e == 1 ? wn[1][q] : wn[2][q]; };
            w_row<P, FC, CC>(ref, m1, Ss, So, Sf, Ts, c, e, jj, of_edge(0), of_edge(1), of_edge(2), -tH * j00,
                             -tH * j01, -tH * j10, -tH * j11, kap, fk, a.W + size_t(j) * NK * N + K, N, wr);
        }
        if constexpr (!FC) {
            __syncthreads();                   // So and Sf have been read
            if (cell && j < M) {
#pragma unroll
                for (int i = 0; i < NP; ++i) So[(j * NP + i) * CC + c] = wr[i];
            }
            __syncthreads();
        }
    }
    if constexpr (FF) {
        // P and Q (f varying over the cell) as float pairs in cell tiles, and the cell's weights (k_ff.cu)
        if constexpr (!FC) {
            constexpr int CP = (NP + 1) / 2;
            for (int idx = t; idx < 2 * NP * CP * CC; idx += kCondThreads) {
                const int cc = idx % CC, pc = idx / CC, i = pc / CP, k0 = 2 * (pc % CP), Kc = blockIdx.x * CC + cc;
                if (Kc >= a.N) continue;
                const double *A = i < NP ? Ps + i * NP * CC : Qs + (i - NP) * NP * CC;
                const float2 v0 = split(A[k0 * CC + cc]);
                const float2 v1 = k0 + 1 < NP ? split(A[(k0 + 1) * CC + cc]) : make_float2(0.f, 0.f);
                a.PQ2[ff_pair_index(size_t(Kc), size_t(pc), size_t(2) * NP * CP)] = make_float4(v0.x, v0.y, v1.x, v1.y);
            }
        }
        if (cell && j == 0) {
            const double jit[4] = {j00, j01, j10, j11};
            float2 *o = a.lgeo + ff_pair_index(size_t(K), 0, kLGeo);
            for (int q = 0; q < 4; ++q) o[size_t(q) * kFFCells] = split(tg * jit[q]);
#pragma unroll
            for (int q = 0; q < 9; ++q) o[size_t(4 + q) * kFFCells] = split(wn[q / 3][q % 3]);
            o[size_t(13) * kFFCells] = split(kap);
            o[size_t(14) * kFFCells] = split(fk);
        }
    }
    if constexpr (!FF && !FC) {
        // Q, P - Q and P + Q for step 3
        for (int idx = t; a.PQ && idx < NP * NP * CC; idx += kCondThreads) {
            const int Kc = blockIdx.x * CC + idx % CC;
            if (Kc >= a.N) continue;
            const double p = Ps[idx], q = Qs[idx];
            double *o = a.PQ + size_t(idx / CC) * N + Kc;
            o[0] = q;
            o[size_t(NP * NP) * N] = p - q;
            o[size_t(2 * NP * NP) * N] = p + q;
        }
    }
    // ---- The h rows of R_M and (FP64 handles that recover by the rows) its velocity rows: the
    // columns of the unit vectors in u_x, u_y and h, spread over all the block's threads.
    // The h columns' h is a column of S^-1 itself.  Where f varies, W_K's entries for r_u too.
    for (int it = t; it < 3 * NP * CC; it += kCondThreads) {
        const int c = it % CC, kap_ = it / CC, comp = kap_ / NP, j = kap_ % NP, K = blockIdx.x * CC + c;
        if (K >= a.N) continue;
        const double j00 = geo[0 * CC + c], j01 = geo[1 * CC + c], j10 = geo[2 * CC + c], j11 = geo[3 * CC + c];
        double wx[NP], wy[NP], h[NP];
        if (comp < 2) {
            double rh[NP];
            const double kap = geo[13 * CC + c], fk = geo[14 * CC + c];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                double p, q;
                if constexpr (FC) {
                    p = i == j ? kap : 0.0;
                    q = i == j ? fk : 0.0;
                } else {
                    p = Ps[(i * NP + j) * CC + c];
                    q = Qs[(i * NP + j) * CC + c];
                }
                wx[i] = comp == 0 ? p : q;
                wy[i] = comp == 0 ? -q : p;
                rh[i] = 0.0;
            }
            add_div<P>(ref, -tH * j00, -tH * j01, -tH * j10, -tH * j11, wx, wy, rh);
            if constexpr (!FF && !FC) {
                double wn[3][3];
#pragma unroll
                for (int e = 0; e < 3; ++e) edge_weights(a, geo, CC, c, K, e, wn[e]);
                w_column<P, CC>(m1, So, c, wn, wx, wy, rh, a.W + size_t(kap_) * N + K, size_t(NK) * N);
            }
            inverse_product<NP, CC>(Ss, c, rh, h);
        } else {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                wx[i] = wy[i] = 0.0;
                h[i] = Ss[(i * NP + j) * CC + c];
            }
        }
        if constexpr (FF) {
            constexpr int CPk = (NK + 1) / 2;
#pragma unroll
            for (int i = 0; i < NP; ++i)
                a.Hr2[2 * ff_pair_index(size_t(K), size_t(i) * CPk + kap_ / 2, size_t(NP) * CPk) + kap_ % 2] = split(h[i]);
        } else {
#pragma unroll
            for (int i = 0; i < NP; ++i) a.Rh[(size_t(i) * NK + kap_) * N + K] = h[i];
            if (a.Ru) {
                subtract_gradient<NP, CC>(Ts, c, h, wx, wy);
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    a.Ru[(size_t(i) * NK + kap_) * N + K] = wx[i];
                    a.Ru[(size_t(NP + i) * NK + kap_) * N + K] = wy[i];
                }
            }
        }
    }
}

// ---------------------------------------------------------------- facet-row assembly
// For facet e with incident (cell, local edge) pairs (K_s, i_s), s = 0, 1, row r
// of the facet (trace node r from the lower to the higher vertex id) is
//   (S x)_{e,r} = sum_c D_e[r][c] x_{e,c} + sum_{s,k} O_{s,k}[r][c] x_{nbr(s,k),c}
// with D_e the sum of both cells' diagonal blocks and O_{s,k} the block of S_{K_s}
// coupling edge i_s to edge (i_s + 1 + k) % 3 (neighbour facet nbr(s,k)).
// Element j = (r*5 + b)*PP + c (b = 0: D_e, b = 1 + 2s + k) of facet e is stored at
// packed_index(j, e, NF, 2) (16-byte groups of two doubles); Dinv = D_e^-1 likewise.
// Padding lanes of the last group are zero.
struct AssembleArgs {
    int N, NF;
    const double *Scell;
    const int32_t *facet_of, *flip, *facet_cell, *facet_edge;
    double *Sval, *Dinv;
    int32_t *nbr;
    int32_t *status;
};

template <int P>
__global__ void assemble_kernel(AssembleArgs a) {
    constexpr int PP = P + 1, M = 3 * PP;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= a.NF) return;
    const size_t NF = a.NF;
    int K[2], I[2], F[2];
    for (int s = 0; s < 2; ++s) {
        K[s] = a.facet_cell[2 * e + s];
        I[s] = a.facet_edge[2 * e + s];
        F[s] = a.flip[3 * K[s] + I[s]];
    }
    double D[PP][PP];
    for (int r = 0; r < PP; ++r)
        for (int c = 0; c < PP; ++c) {
            double v = 0.0;
            for (int s = 0; s < 2; ++s) {
                const int lr = I[s] * PP + (F[s] ? P - r : r);
                const int lc = I[s] * PP + (F[s] ? P - c : c);
                v += a.Scell[size_t(K[s]) * M * M + lr * M + lc];
            }
            D[r][c] = v;
            a.Sval[packed_index((r * 5 + 0) * PP + c, e, NF, 2)] = v;
        }
    for (int s = 0; s < 2; ++s)
        for (int k = 0; k < 2; ++k) {
            const int b = 1 + 2 * s + k;
            const int i2 = (I[s] + 1 + k) % 3;
            const int f2 = a.flip[3 * K[s] + i2];
            a.nbr[size_t(b - 1) * NF + e] = a.facet_of[3 * K[s] + i2];
            for (int r = 0; r < PP; ++r) {
                const int lr = I[s] * PP + (F[s] ? P - r : r);
                for (int c = 0; c < PP; ++c) {
                    const int lc = i2 * PP + (f2 ? P - c : c);
                    a.Sval[packed_index((r * 5 + b) * PP + c, e, NF, 2)] = a.Scell[size_t(K[s]) * M * M + lr * M + lc];
                }
            }
        }
    // invert D_e (Gauss-Jordan with partial pivoting, in registers)
    double Inv[PP][PP];
    for (int r = 0; r < PP; ++r)
        for (int c = 0; c < PP; ++c) Inv[r][c] = (r == c) ? 1.0 : 0.0;
    bool singular = false;
    for (int k = 0; k < PP; ++k) {
        int pr = k;
        double best = fabs(D[k][k]);
        for (int r = k + 1; r < PP; ++r)
            if (fabs(D[r][k]) > best) { best = fabs(D[r][k]); pr = r; }
        if (!(best > 1e-300)) { singular = true; break; }
        if (pr != k)
            for (int c = 0; c < PP; ++c) {
                double t = D[k][c]; D[k][c] = D[pr][c]; D[pr][c] = t;
                t = Inv[k][c]; Inv[k][c] = Inv[pr][c]; Inv[pr][c] = t;
            }
        const double pinv = 1.0 / D[k][k];
        for (int c = 0; c < PP; ++c) { D[k][c] *= pinv; Inv[k][c] *= pinv; }
        for (int r = 0; r < PP; ++r) {
            if (r == k) continue;
            const double f = D[r][k];
            for (int c = 0; c < PP; ++c) { D[r][c] -= f * D[k][c]; Inv[r][c] -= f * Inv[k][c]; }
        }
    }
    if (singular) atomicOr(a.status, 2);
    for (int r = 0; r < PP; ++r)
        for (int c = 0; c < PP; ++c) a.Dinv[packed_index(r * PP + c, e, NF, 2)] = Inv[r][c];
    if ((5 * PP * PP) % 2) a.Sval[packed_index(5 * PP * PP, e, NF, 2)] = 0.0;
    if ((PP * PP) % 2) a.Dinv[packed_index(PP * PP, e, NF, 2)] = 0.0;
}

// ---------------------------------------------------------------- P1 level operator
// The coarse problem obtained, as in Sec. 4.4 (Eq. coarse_problem_upwind), by
// eliminating u from the time-implicit continuum equations, here with the
// Coriolis term implicit: u = (I - tau f J)(r_u - tau g grad h)/(1 + tau^2 f^2),
// hence per cell (f_K the cell mean of f, kappa_K = 1/(1 + tau^2 f_K^2))
//   A = [ (phi,psi) + tau^2 g H kappa_K ((grad phi, grad psi) - tau f_K (J grad phi, grad psi)) ] / tau,
// divided by tau to match the scale of the trace operator on smooth traces.
// rotating = 0 drops f (the form printed in the paper).  Every CSR entry sums
// its contributions in a fixed (cell) order.
//
// One launch forms every level's values, inverse diagonal and their FP32 copies, a thread
// per ELL slot.  What it takes is the latency of one slot's chain (contribution list,
// element entries, sum), so the levels run side by side and the division by tau is left to
// the end: r = 5, five levels, 28 us for all of it instead of 120 in twenty launches.
constexpr int kP1Levels = 12;
struct P1Levels {
    int n;
    int start[kP1Levels + 1];               // first thread of each level
    struct Level {
        int width;
        const int32_t *cptr, *contrib, *diag;
        const double *elem, *fK;
        double *A, *dinv;
        float *A32, *dinv32;                // null in FP64
    } l[kP1Levels];
};
__global__ void __launch_bounds__(256) p1_levels_kernel(const __grid_constant__ P1Levels m, double tau, double gH,
                                                        int rotating) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m.start[m.n]) return;
    int i = 0;
    while (t >= m.start[i + 1]) ++i;
    const P1Levels::Level &L = m.l[i];
    const int q = t - m.start[i], k1 = L.cptr[q + 1];
    const double t2 = tau * tau, t2g = t2 * gH;
    double acc = 0.0;
    for (int k = L.cptr[q]; k < k1; ++k) {
        const int code = L.contrib[k], K = code / 9, ab = code % 9;
        const double *el = L.elem + size_t(K) * 27;
        const double e0 = el[ab], e1 = el[9 + ab];
        if (rotating) {
            const double f = L.fK[K];
            acc += e0 + t2g * reciprocal(fma(t2 * f, f, 1.0)) * (e1 - tau * f * el[18 + ab]);
        } else {
            acc += e0 + t2g * e1;
        }
    }
    acc /= tau;
    L.A[q] = acc;
    if (L.A32) L.A32[q] = to_float(acc);
    const int v = q / L.width;
    if (L.diag[v] == q) {
        const double r = 1.0 / acc;
        L.dinv[v] = r;
        if (L.dinv32) L.dinv32[v] = to_float(r);
    }
}

// dense copy of a padded ELL matrix (kInvSmem < n <= 1024; unused slots add 0 to the
// diagonal), then Gauss-Jordan inverse with partial pivoting, by one CTA up to n = 256.
__global__ void ell_to_dense_kernel(int n, int width, const int32_t *col, const double *A, double *D) {
    const int r = blockIdx.x;
    for (int c = threadIdx.x; c < n; c += blockDim.x) D[size_t(r) * n + c] = 0.0;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int q = 0; q < width; ++q) D[size_t(r) * n + col[size_t(r) * width + q]] += A[size_t(r) * width + q];
}

// The inverse of a small ELL matrix (n <= kInvSmem) by in-place Gauss-Jordan elimination
// with partial pivoting in the shared memory of one CTA, each element with the arithmetic
// of the kernels below, so that all give the same inverse bit for bit.  Bound by the chain
// of n steps, three barriers each: 80 us for 42 vertices, 52 for 36, instead of 160 and 127
// with matrix and inverse in global memory and a tree of 1024 threads per pivot.
constexpr int kInvSmem = 160;
constexpr int kInvThreads = 256;             // fits an SM beside the condensation's blocks
__global__ void __launch_bounds__(kInvThreads) ell_inverse_kernel(int n, int width, const int32_t *__restrict__ col,
                                                                  const double *__restrict__ Ae,
                                                                  double *__restrict__ inv, int32_t *status) {
    extern __shared__ double A[];              // [n][n], the pivot row, the pivot column
    double *row = A + size_t(n) * n, *fac = row + n;
    __shared__ int piv[kInvSmem];
    const int tid = threadIdx.x, lane = tid & 31;
    for (int k = tid; k < n * n; k += kInvThreads) A[k] = 0.0;
    __syncthreads();
    if (tid < n)
        for (int q = 0; q < width; ++q) A[tid * n + col[size_t(tid) * width + q]] += Ae[size_t(tid) * width + q];
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (tid < 32) {
            // largest magnitude (as bits, which order alike), then the lowest row; a NaN never wins
            long long best = -1;
            int p = k;
            for (int r = k + lane; r < n; r += 32) {
                const long long v = __double_as_longlong(A[r * n + k]) & 0x7fffffffffffffffll;
                if (v <= 0x7ff0000000000000ll && v > best) {
                    best = v;
                    p = r;
                }
            }
            for (int off = 16; off > 0; off >>= 1) {
                const long long v = __shfl_xor_sync(0xffffffffu, best, off);
                const int r = __shfl_xor_sync(0xffffffffu, p, off);
                if (v > best || (v == best && r < p)) {
                    best = v;
                    p = r;
                }
            }
            if (lane == 0) {
                piv[k] = p;
                if (best < 0 || !(__longlong_as_double(best) > 1e-300)) atomicOr(status, 4);
            }
        }
        __syncthreads();
        const int p = piv[k];
        if (tid < n) {
            // the pivot row scaled, row k in its place; the factors of the other rows
            const int c = tid;
            const double pinv = 1.0 / A[p * n + k], akc = A[k * n + c], apc = A[p * n + c];
            row[c] = c == k ? pinv : apc * pinv;
            fac[c] = c == p ? A[k * n + k] : A[c * n + k];
            if (p != k && c != k) A[p * n + c] = akc;      // (column k is not read again)
        }
        __syncthreads();
        for (int idx = tid; idx < n * n; idx += kInvThreads) {
            const int r = idx / n, c = idx - r * n;
            A[idx] = r == k ? row[c] : fma(-fac[r], row[c], c == k ? 0.0 : A[idx]);
        }
        __syncthreads();
    }
    // the row swaps, undone on the columns in reverse order: column j goes to place q
    for (int idx = tid; idx < n * n; idx += kInvThreads) {
        const int r = idx / n, j = idx - r * n;
        int q = j;
        for (int k = n - 1; k >= 0; --k) {
            const int p = piv[k];
            q = q == k ? p : q == p ? k : q;
        }
        inv[r * n + q] = A[idx];
    }
}

__global__ void dense_inverse_kernel(int n, double *Aw, double *inv, int32_t *status) {
    // Aw: working copy [n][n], destroyed; inv: output [n][n]
    __shared__ int piv_row;
    __shared__ double red_v[1024];
    __shared__ int red_i[1024];
    const int tid = threadIdx.x;
    for (int idx = tid; idx < n * n; idx += blockDim.x) inv[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        double best = -1.0;
        int bi = k;
        for (int r = k + tid; r < n; r += blockDim.x) {
            double v = fabs(Aw[size_t(r) * n + k]);
            if (v > best) { best = v; bi = r; }
        }
        red_v[tid] = best;
        red_i[tid] = bi;
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if (tid < s && red_v[tid + s] > red_v[tid]) { red_v[tid] = red_v[tid + s]; red_i[tid] = red_i[tid + s]; }
            __syncthreads();
        }
        if (tid == 0) {
            piv_row = red_i[0];
            if (!(red_v[0] > 1e-300)) atomicOr(status, 4);
        }
        __syncthreads();
        const int pr = piv_row;
        if (pr != k)
            for (int c = tid; c < n; c += blockDim.x) {
                double t = Aw[size_t(k) * n + c]; Aw[size_t(k) * n + c] = Aw[size_t(pr) * n + c]; Aw[size_t(pr) * n + c] = t;
                t = inv[size_t(k) * n + c]; inv[size_t(k) * n + c] = inv[size_t(pr) * n + c]; inv[size_t(pr) * n + c] = t;
            }
        __syncthreads();
        const double pinv = 1.0 / Aw[size_t(k) * n + k];
        __syncthreads();
        for (int c = tid; c < n; c += blockDim.x) {
            Aw[size_t(k) * n + c] *= pinv;
            inv[size_t(k) * n + c] *= pinv;
        }
        __syncthreads();
        for (int idx = tid; idx < n * n; idx += blockDim.x) {
            const int r = idx / n, c = idx % n;
            if (r == k) continue;
            const double f = Aw[size_t(r) * n + k];
            if (c != k) Aw[size_t(r) * n + c] -= f * Aw[size_t(k) * n + c];
            inv[size_t(r) * n + c] -= f * inv[size_t(k) * n + c];
        }
        __syncthreads();
        for (int r = tid; r < n; r += blockDim.x)
            if (r != k) Aw[size_t(r) * n + k] = 0.0;
        __syncthreads();
    }
}

// The same elimination over many blocks, for coarsest levels too large for
// one CTA: step k is two launches, the pivot (search as above, row swap,
// scaling of row k, and a copy of column k as the row factors) and the
// update of every other row, each element with the single-CTA kernel's
// arithmetic, so that both give the same inverse bit for bit.
__global__ void gj_pivot_kernel(int n, int k, double *Aw, double *inv, double *fac, int32_t *status) {
    __shared__ int piv_row;
    __shared__ double red_v[1024];
    __shared__ int red_i[1024];
    const int tid = threadIdx.x;
    double best = -1.0;
    int bi = k;
    for (int r = k + tid; r < n; r += blockDim.x) {
        const double v = fabs(Aw[size_t(r) * n + k]);
        if (v > best) { best = v; bi = r; }
    }
    red_v[tid] = best;
    red_i[tid] = bi;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (tid < s && red_v[tid + s] > red_v[tid]) { red_v[tid] = red_v[tid + s]; red_i[tid] = red_i[tid + s]; }
        __syncthreads();
    }
    if (tid == 0) {
        piv_row = red_i[0];
        if (!(red_v[0] > 1e-300)) atomicOr(status, 4);
    }
    __syncthreads();
    const int pr = piv_row;
    if (pr != k)
        for (int c = tid; c < n; c += blockDim.x) {
            double t = Aw[size_t(k) * n + c]; Aw[size_t(k) * n + c] = Aw[size_t(pr) * n + c]; Aw[size_t(pr) * n + c] = t;
            t = inv[size_t(k) * n + c]; inv[size_t(k) * n + c] = inv[size_t(pr) * n + c]; inv[size_t(pr) * n + c] = t;
        }
    __syncthreads();
    const double pinv = 1.0 / Aw[size_t(k) * n + k];
    __syncthreads();
    for (int c = tid; c < n; c += blockDim.x) {
        Aw[size_t(k) * n + c] *= pinv;
        inv[size_t(k) * n + c] *= pinv;
    }
    for (int r = tid; r < n; r += blockDim.x) fac[r] = Aw[size_t(r) * n + k];
}

// (columns left of the pivot of the working copy are skipped: their row-k
// entries are exact zeros, so the single-CTA update leaves them unchanged)
__global__ void gj_update_kernel(int n, int k, double *Aw, double *inv, const double *fac) {
    const size_t idx = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= size_t(n) * n) return;
    const int r = int(idx / n), c = int(idx % n);
    if (r == k) return;
    const double f = fac[r];
    if (c > k) Aw[size_t(r) * n + c] -= f * Aw[size_t(k) * n + c];
    else if (c == k) Aw[size_t(r) * n + k] = 0.0;
    inv[size_t(r) * n + c] -= f * inv[size_t(k) * n + c];
}

__global__ void identity_kernel(int n, double *inv) {
    const size_t idx = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx < size_t(n) * n) inv[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
}

__global__ void to_f32_kernel(const double *x, float *y, size_t n) {
    size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n) y[i] = to_float(x[i]);
}

template <int P, bool FC, bool FF>
cudaError_t condense_nodal_p(hdg_handle *h) {
    constexpr size_t smem = sizeof(double) * CondSmem<P, FC>::total;
    auto k = &condense_nodal_kernel<P, FC, FF>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    NodalArgs a;
    a.N = h->N; a.tau = h->prm.tau; a.g = h->prm.g; a.H = h->prm.H; a.ts = h->tau_s;
    a.nref = h->d_nref; a.M1 = h->d_ref + ref_offsets(P).M1; a.X = h->d_X; a.fcell = h->d_fcell;
    a.Xb = h->d_Xb; a.W = h->d_W; a.Scell = h->d_Scell; a.status = h->d_status;
    a.Rh = FF ? nullptr : h->d_Rm + size_t(rm_offsets(P, FC, h->rec_rows).h) * h->N;
    a.Ru = h->rec_rows ? h->d_Rm : nullptr;
    a.PQ = h->rec_rows ? nullptr : h->d_Rm;
    a.Xb2 = h->d_Xb2; a.Hr2 = h->d_Hr2; a.lgeo = h->d_lgeo; a.PQ2 = reinterpret_cast<float4 *>(h->d_PQ2);
    k<<<(h->N + kCondCells<P> - 1) / kCondCells<P>, kCondThreads, smem, h->stream>>>(a);
    return cudaGetLastError();
}
template <int P>
cudaError_t condense_p(hdg_handle *h) {
    if (mode_ff(h->prm)) return h->f_const ? condense_nodal_p<P, true, true>(h) : condense_nodal_p<P, false, true>(h);
    return h->f_const ? condense_nodal_p<P, true, false>(h) : condense_nodal_p<P, false, false>(h);
}

template <int P>
cudaError_t assemble_p(hdg_handle *h) {
    AssembleArgs a;
    a.N = h->N; a.NF = h->NF; a.Scell = h->d_Scell;
    a.facet_of = h->d_facet_of; a.flip = h->d_flip; a.facet_cell = h->d_facet_cell; a.facet_edge = h->d_facet_edge;
    a.Sval = h->d_Sval; a.Dinv = h->d_Dinv; a.nbr = h->d_nbr; a.status = h->d_status;
    assemble_kernel<P><<<(h->NF + 127) / 128, 128, 0, h->stream>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_condense(hdg_handle *h) {
    switch (h->p) {
        case 1: return condense_p<1>(h);
        case 2: return condense_p<2>(h);
        case 3: return condense_p<3>(h);
        case 4: return condense_p<4>(h);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_assemble(hdg_handle *h) {
    switch (h->p) {
        case 1: return assemble_p<1>(h);
        case 2: return assemble_p<2>(h);
        case 3: return assemble_p<3>(h);
        case 4: return assemble_p<4>(h);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_p1_levels(hdg_handle *h, double tau, double gH, int rotating) {
    for (size_t l0 = 0; l0 < h->lev.size(); l0 += kP1Levels) {
        P1Levels m = {};
        m.n = int(std::min(h->lev.size() - l0, size_t(kP1Levels)));
        for (int i = 0; i < m.n; ++i) {
            const DevLevel &L = h->lev[l0 + size_t(i)];
            m.start[i + 1] = m.start[i] + L.nnz;
            m.l[i] = {L.width, L.contrib_ptr, L.contrib, L.diag, L.elem, L.fK, L.A, L.dinv, L.A32, L.dinv32};
        }
        p1_levels_kernel<<<unsigned(m.start[m.n] + 255) / 256, 256, 0, h->stream>>>(m, tau, gH, rotating);
    }
    return cudaGetLastError();
}

cudaError_t launch_dense_inverse(hdg_handle *h, const DevLevel &L, double *work, double *inv, int n) {
    if (n <= kInvSmem) {
        const size_t smem = sizeof(double) * size_t(n) * size_t(n + 2);
        cudaError_t e = cudaFuncSetAttribute(ell_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             int(sizeof(double) * kInvSmem * (kInvSmem + 2)));
        if (e != cudaSuccess) return e;
        ell_inverse_kernel<<<1, kInvThreads, smem, h->stream>>>(n, L.width, L.col, L.A, inv, h->d_status);
        return cudaGetLastError();
    }
    ell_to_dense_kernel<<<n, 128, 0, h->stream>>>(n, L.width, L.col, L.A, work);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (n <= 256) {
        dense_inverse_kernel<<<1, 1024, 0, h->stream>>>(n, work, inv, h->d_status);
        return cudaGetLastError();
    }
    // larger coarsest levels: one pivot and one update launch per column, the
    // row factors of each column in their own array
    double *fac = h->d_coarse_fac;
    if (!fac) return cudaErrorInvalidValue;
    const size_t nn = size_t(n) * n;
    const unsigned nb = unsigned((nn + 255) / 256);
    identity_kernel<<<nb, 256, 0, h->stream>>>(n, inv);
    for (int k = 0; k < n; ++k) {
        gj_pivot_kernel<<<1, 1024, 0, h->stream>>>(n, k, work, inv, fac, h->d_status);
        gj_update_kernel<<<nb, 256, 0, h->stream>>>(n, k, work, inv, fac);
    }
    return cudaGetLastError();
}

cudaError_t launch_to_f32(const double *x, float *y, size_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    to_f32_kernel<<<unsigned((n + 255) / 256), 256, 0, s>>>(x, y, n);
    return cudaGetLastError();
}

}  // namespace hdg
