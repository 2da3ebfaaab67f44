// IMEX time stepping around the implicit solve (Sec. 3.3, Eqs. theta_method,
// IMEX_HDG_I and IMEX_HDG_II; tableaux of Sec. 5.1).
//
// The semi-discrete system is M dq/dt = N(q) + L(q): L holds the gravity-wave
// terms with the upwind stabilisation (taken implicitly), N the Coriolis term
// (taken explicitly, as in the paper).  Everything here works on nodal
// function values (the caller's u [N][2][n_p], h [N][n_p] layout), so each
// mass matrix is applied through its inverse per cell:
//   n~(q) = M^-1 N(q),  l~(q) = M^-1 L(q).
// An implicit stage M Q - a~_ii dt L(Q) = M r is the hot path's solve with
// f = 0 and tau = a~_ii dt, right-hand-side function r (hdg_solve_dev +
// hdg_recover_dev).  L is evaluated from the DG state: the trace on each facet
// is the upwind value lambda = {h} + H / (2 tau_s) (u_1.n_1 + u_2.n_2) (the
// HDG transmission condition solved pointwise; every trace is in P^p(e)), and
// per cell, in the integrated-by-parts form of the library's condensation,
//   L_u(q) . w  = g (h, div w) - g <lambda, w.n>_dK
//   L_h(q) psi  = -H (div u, psi) - tau_s <h - lambda, psi>_dK
//   N_u(q) . w  = -(f u_perp, w),  N_h = 0,   u_perp = (-u_y, u_x).
#include "common.h"

#include <algorithm>
#include <cmath>

namespace hdg {
namespace {

inline unsigned nblocks(size_t n, int bs) { return unsigned((n + bs - 1) / bs); }

// tangent of edge i (from local vertex (i+1)%3 to (i+2)%3) of a cell with
// local vertices x[6]; (ty, -tx) is its outward normal times its length
__device__ __forceinline__ void edge_tangent(const double *x, int i, double &tx, double &ty) {
    const int v1 = (i + 1) % 3, v2 = (i + 2) % 3;
    tx = x[2 * v2] - x[2 * v1];
    ty = x[2 * v2 + 1] - x[2 * v1 + 1];
}

// lambda at the p+1 trace nodes of every facet (internal layout [PP][NF]);
// c = H / (2 tau_s)
template <int P>
__global__ void upwind_trace_kernel(int NF, const int32_t *__restrict__ fcell, const int32_t *__restrict__ fedge,
                                    const int32_t *__restrict__ flip, const double *__restrict__ X,
                                    const double *__restrict__ u, const double *__restrict__ h, double c,
                                    double *__restrict__ lam) {
    constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    double v[PP];
#pragma unroll
    for (int r = 0; r < PP; ++r) v[r] = 0.0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int K = fcell[2 * e + s], i = fedge[2 * e + s], fl = flip[3 * K + i];
        double x[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) x[k] = X[size_t(K) * 6 + k];
        double tx, ty;
        edge_tangent(x, i, tx, ty);
        const double w = c / sqrt(tx * tx + ty * ty), wx = w * ty, wy = -w * tx;
#pragma unroll
        for (int r = 0; r < PP; ++r) {
            const int node = edge_cell_node(P, i, fl ? P - r : r);
            const double hv = h[size_t(K) * NP + node];
            v[r] = fma(wx, u[size_t(K) * 2 * NP + node], fma(wy, u[size_t(K) * 2 * NP + NP + node], fma(0.5, hv, v[r])));
        }
    }
#pragma unroll
    for (int r = 0; r < PP; ++r) lam[size_t(r) * NF + e] = v[r];
}

struct RateArgs {
    int N, NF;
    double g, H, ts;
    const double *nref;      // packed nodal reference matrices
    const double *X;         // [N][3][2]
    const double *fcell;     // [N][3] Coriolis at the cell's vertices (P1), or null
    const int32_t *facet_of, *flip;
    const double *lam;       // [PP][NF]
    const double *u, *h;     // state
    double *nu, *nh;         // M^-1 N(q): u part (N kernels), h part (zero, when given)
    double *lu, *lh;         // M^-1 L(q) (L kernels)
};

// The rates of 64 cells per block, one thread per cell, in function space (every
// matrix of the reference element multiplied by M_ref^-1 on the host, so no mass
// solve is left and |det J| drops out).  L is integrated by parts to the strong
// form, whose facet terms all act on the jump d = h - lambda: with
// s_i = lift_i d_i / |det J| (t the edge tangent, J^-T = j),
//   l~_u = -g grad h + g sum_i (t_y, -t_x)_i s_i,
//   l~_h = -H div u - tau_s sum_i |e_i| s_i,
// div u through the contravariant components (two matrix products, not four),
// and n~ through f's P1 form f_0 + (f_1 - f_0) L_1 + (f_2 - f_0) L_2.
// What bounds it is the FP64 pipe (1.05 TFLOP/s measured): about 570 FMAs per cell
// for L and 430 for N at p = 3 (no derivative entry that vanishes is multiplied)
// against about 3,500 FP64 operations in the weak form with a mass solve per
// field (554 us per launch on the r = 6 sphere, 81,920 cells, p = 3).  An ARS2
// step there went from 4,596 to 3,250 us with these rates, the first stage's
// unused l~ left out and the combinations below.  Cells are staged through shared memory
// (odd stride: no bank conflicts) so that global reads and writes coalesce.
constexpr int kRateCells = 64;
template <int P, bool L, bool N>
__global__ void __launch_bounds__(kRateCells) imex_rates_kernel(RateArgs a) {
    constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2, NK = 3 * NP, LD = NK | 1;
    constexpr NodalOffsets O = nodal_offsets(P);
    __shared__ double ref[O.Wx];            // all but the weak derivatives
    __shared__ double sS[kRateCells * LD];
    const int t = threadIdx.x;
    const int K0 = blockIdx.x * kRateCells, nc = min(kRateCells, a.N - K0);
    for (int k = t; k < O.Wx; k += kRateCells) ref[k] = a.nref[k];
    for (int k = t; k < nc * 2 * NP; k += kRateCells) sS[(k / (2 * NP)) * LD + k % (2 * NP)] = a.u[size_t(K0) * 2 * NP + k];
    if (L)
        for (int k = t; k < nc * NP; k += kRateCells) sS[(k / NP) * LD + 2 * NP + k % NP] = a.h[size_t(K0) * NP + k];
    __syncthreads();
    const int K = K0 + t;
    const bool on = t < nc;
    double *q = sS + t * LD;                  // this thread's cell: the state, then its rates
    double ux[NP], uy[NP];
    if (on) {
#pragma unroll
        for (int b = 0; b < NP; ++b) {
            ux[b] = q[b];
            uy[b] = q[NP + b];
        }
    }
    if constexpr (L) {
        if (on) {
            double x[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) x[k] = a.X[size_t(K) * 6 + k];
            const double J00 = x[2] - x[0], J01 = x[4] - x[0], J10 = x[3] - x[1], J11 = x[5] - x[1];
            const double s = 1.0 / (J00 * J11 - J01 * J10);
            // J^-T: d/dx = j00 d/dxi + j01 d/deta, d/dy = j10 d/dxi + j11 d/deta
            const double j00 = J11 * s, j01 = -J10 * s, j10 = -J01 * s, j11 = J00 * s;
            double hh[NP], d[3][PP], wx[3], wy[3], wh[3];
#pragma unroll
            for (int b = 0; b < NP; ++b) hh[b] = q[2 * NP + b];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                double tx, ty;
                edge_tangent(x, i, tx, ty);
                wx[i] = a.g * ty;
                wy[i] = -a.g * tx;
                wh[i] = -a.ts * sqrt(tx * tx + ty * ty);
                const int f = a.facet_of[3 * K + i], fl = a.flip[3 * K + i];
#pragma unroll
                for (int j = 0; j < PP; ++j)
                    d[i][j] = s * (hh[edge_cell_node(P, i, j)] - a.lam[size_t(fl ? P - j : j) * a.NF + f]);
            }
            const double g00 = -a.g * j00, g01 = -a.g * j01, g10 = -a.g * j10, g11 = -a.g * j11;
            // the contravariant velocity times -H
            double c1[NP], c2[NP];
#pragma unroll
            for (int b = 0; b < NP; ++b) {
                c1[b] = -a.H * fma(j00, ux[b], j10 * uy[b]);
                c2[b] = -a.H * fma(j01, ux[b], j11 * uy[b]);
            }
            static_for<NP>([&](auto ia_) {
                constexpr int ia = decltype(ia_)::value;
                double hx = 0.0, hy = 0.0, lh = 0.0;
                static_for<NP>([&](auto ib_) {
                    constexpr int ib = decltype(ib_)::value;
                    if constexpr (nodal_dx_nonzero(P, ia, ib)) {
                        const double m = ref[O.Dx + ia * NP + ib];
                        hx = fma(m, hh[ib], hx);
                        lh = fma(m, c1[ib], lh);
                    }
                    if constexpr (nodal_dy_nonzero(P, ia, ib)) {
                        const double m = ref[O.Dy + ia * NP + ib];
                        hy = fma(m, hh[ib], hy);
                        lh = fma(m, c2[ib], lh);
                    }
                });
                double lx = fma(g00, hx, g01 * hy), ly = fma(g10, hx, g11 * hy);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    double si = 0.0;
#pragma unroll
                    for (int j = 0; j < PP; ++j) si = fma(ref[O.lift + (i * NP + ia) * PP + j], d[i][j], si);
                    lx = fma(wx[i], si, lx);
                    ly = fma(wy[i], si, ly);
                    lh = fma(wh[i], si, lh);
                }
                q[ia] = lx;
                q[NP + ia] = ly;
                q[2 * NP + ia] = lh;
            });
        }
        __syncthreads();
        for (int k = t; k < nc * 2 * NP; k += kRateCells)
            a.lu[size_t(K0) * 2 * NP + k] = sS[(k / (2 * NP)) * LD + k % (2 * NP)];
        for (int k = t; k < nc * NP; k += kRateCells) a.lh[size_t(K0) * NP + k] = sS[(k / NP) * LD + 2 * NP + k % NP];
        if constexpr (N) __syncthreads();
    }
    if constexpr (N) {
        if (on) {
            // (n~_x, n~_y) = (F u_y, -F u_x), F the projected multiplication by f
            const double f0 = a.fcell[size_t(K) * 3];
            const double f1 = a.fcell[size_t(K) * 3 + 1] - f0, f2 = a.fcell[size_t(K) * 3 + 2] - f0;
#pragma unroll
            for (int ia = 0; ia < NP; ++ia) {
                double nx = f0 * uy[ia], ny = f0 * ux[ia];
#pragma unroll
                for (int ib = 0; ib < NP; ++ib) {
                    const double m = fma(f1, ref[O.ML1 + ia * NP + ib], f2 * ref[O.ML2 + ia * NP + ib]);
                    nx = fma(m, uy[ib], nx);
                    ny = fma(m, ux[ib], ny);
                }
                q[ia] = nx;
                q[NP + ia] = -ny;
            }
        }
        __syncthreads();
        for (int k = t; k < nc * 2 * NP; k += kRateCells)
            a.nu[size_t(K0) * 2 * NP + k] = sS[(k / (2 * NP)) * LD + k % (2 * NP)];
        if (a.nh)
            for (int k = t; k < nc * NP; k += kRateCells) a.nh[size_t(K0) * NP + k] = 0.0;
    }
}

// out = q0 + dt sum_j c_j x_j over a whole state (u part of nu entries, then h
// part; q0 and out in two pieces each, which may be the caller's); terms j < kn
// are rates n~, whose h part is zero and not read.  Only the terms with a
// non-zero coefficient are passed.  Four entries per thread, a block width
// apart, so that their loads overlap.
struct Combo {
    int k = 0, kn = 0;
    double c[2 * kImexMaxStages];
    const double *x[2 * kImexMaxStages];
};
constexpr int kCombU = 4;
__global__ void __launch_bounds__(256) imex_combine_kernel(size_t nu, size_t n, const double *q0u, const double *q0h,
                                                           Combo c, double dt, double *outu, double *outh) {
    const size_t i0 = size_t(blockIdx.x) * blockDim.x * kCombU + threadIdx.x;
    double q[kCombU], acc[kCombU];
#pragma unroll
    for (int u = 0; u < kCombU; ++u) {
        const size_t i = i0 + size_t(u) * blockDim.x;
        q[u] = i < nu ? q0u[i] : i < n ? q0h[i - nu] : 0.0;
        acc[u] = 0.0;
    }
    for (int j = 0; j < c.k; ++j) {
        const double cj = c.c[j];
        const double *x = c.x[j];
        const size_t m = j < c.kn ? nu : n;
#pragma unroll
        for (int u = 0; u < kCombU; ++u) {
            const size_t i = i0 + size_t(u) * blockDim.x;
            if (i < m) acc[u] = fma(cj, x[i], acc[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < kCombU; ++u) {
        const size_t i = i0 + size_t(u) * blockDim.x;
        const double v = fma(dt, acc[u], q[u]);
        if (i < nu) outu[i] = v;
        else if (i < n) outh[i - nu] = v;
    }
}

// Butcher tableaux (explicit a, implicit a~, weights b, b~) of Sec. 5.1
struct Tableau {
    int s;
    double a[5][5], at[5][5], b[5], bt[5];
};

Tableau tableau(int scheme, double theta) {
    Tableau T{};
    if (scheme == HDG_IMEX_THETA) {
        // M q1 = M q0 + dt (N(q0) + (1 - theta) L(q0) + theta L(q1)) as a
        // two-stage method: Q_1 = q0 (explicit), Q_2 implicit with a~_22 = theta
        T.s = 2;
        T.a[1][0] = 1.0;
        T.at[1][0] = 1.0 - theta;
        T.at[1][1] = theta;
        T.b[0] = 1.0;
        T.bt[0] = 1.0 - theta;
        T.bt[1] = theta;
    } else if (scheme == HDG_IMEX_ARS2) {
        const double g = 1.0 - 1.0 / std::sqrt(2.0), d = -2.0 * std::sqrt(2.0) / 3.0;
        T.s = 3;
        T.a[1][0] = g;
        T.a[2][0] = d; T.a[2][1] = 1.0 - d;
        T.at[1][1] = g;
        T.at[2][1] = 1.0 - g; T.at[2][2] = g;
        T.b[1] = 1.0 - g; T.b[2] = g;
        T.bt[1] = 1.0 - g; T.bt[2] = g;
    } else if (scheme == HDG_IMEX_SSP2) {
        T.s = 3;
        T.a[2][1] = 1.0;
        T.at[0][0] = 0.5;
        T.at[1][0] = -0.5; T.at[1][1] = 0.5;
        T.at[2][1] = 0.5; T.at[2][2] = 0.5;
        T.b[1] = 0.5; T.b[2] = 0.5;
        T.bt[1] = 0.5; T.bt[2] = 0.5;
    } else {   // ARS3(4,4,3)
        T.s = 5;
        const double A[5][5] = {{0, 0, 0, 0, 0}, {0.5, 0, 0, 0, 0}, {11.0 / 18, 1.0 / 18, 0, 0, 0},
                                {5.0 / 6, -5.0 / 6, 0.5, 0, 0}, {0.25, 1.75, 0.75, -1.75, 0}};
        const double At[5][5] = {{0, 0, 0, 0, 0}, {0, 0.5, 0, 0, 0}, {0, 1.0 / 6, 0.5, 0, 0},
                                 {0, -0.5, 0.5, 0.5, 0}, {0, 1.5, -1.5, 0.5, 0.5}};
        for (int i = 0; i < 5; ++i)
            for (int j = 0; j < 5; ++j) {
                T.a[i][j] = A[i][j];
                T.at[i][j] = At[i][j];
            }
        const double b[5] = {0.25, 1.75, 0.75, -1.75, 0}, bt[5] = {0, 1.5, -1.5, 0.5, 0.5};
        for (int i = 0; i < 5; ++i) {
            T.b[i] = b[i];
            T.bt[i] = bt[i];
        }
    }
    return T;
}

}  // namespace

cudaError_t launch_imex_rates(hdg_handle *h, const double *u, const double *hh, double *nu, double *nh, double *lu,
                              double *lh) {
    Imex &I = h->imex;
    RateArgs a{h->N, h->NF, h->prm.g, h->prm.H, h->tau_s, h->d_nref, h->d_X, I.fcell, h->d_facet_of,
               h->d_flip, I.lam, u, hh, nu, nh, lu, lh};
    const unsigned nb = nblocks(h->N, kRateCells);
    if (!lu) {
        HDG_DISPATCH_P(h->p, (imex_rates_kernel<P, false, true><<<nb, kRateCells, 0, h->stream>>>(a)));
        return cudaGetLastError();
    }
    HDG_DISPATCH_P(h->p, (upwind_trace_kernel<P><<<nblocks(h->NF, 256), 256, 0, h->stream>>>(
                             h->NF, h->d_facet_cell, h->d_facet_edge, h->d_flip, h->d_X, u, hh,
                             h->prm.H / (2.0 * h->tau_s), I.lam)));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (nu) {
        HDG_DISPATCH_P(h->p, (imex_rates_kernel<P, true, true><<<nb, kRateCells, 0, h->stream>>>(a)));
    } else {
        HDG_DISPATCH_P(h->p, (imex_rates_kernel<P, true, false><<<nb, kRateCells, 0, h->stream>>>(a)));
    }
    return cudaGetLastError();
}

}  // namespace hdg

using namespace hdg;

namespace {

int imex_fail(hdg_handle *h, int code, const std::string &msg) {
    h->err = msg;
    return code;
}

void imex_free(Imex &I) {
    for (double **p : {&I.fcell, &I.lam, &I.lam_out, &I.buf})
        if (*p) {
            cudaFree(*p);
            *p = nullptr;
        }
    I.ready = false;
}

}  // namespace

void hdg::imex_release(hdg_handle *h) { imex_free(h->imex); }

extern "C" int hdg_imex_init(hdg_handle *h, const double *f_vertex) {
    if (!h) return HDG_EINVAL;
    if (h->prm.flux != 0)
        return imex_fail(h, HDG_EINVAL, "hdg_imex_init: the IMEX stages use the upwind solver");
    if (h->has_f)
        return imex_fail(h, HDG_EINVAL,
                         "hdg_imex_init: the implicit stages have no Coriolis term; set the handle up with "
                         "f_vertex = NULL and pass the Coriolis field here");
    Imex &I = h->imex;
    imex_free(I);
    const size_t N = h->N, np = h->np, nq = N * 3 * np;
    std::vector<double> fcell(N * 3, 0.0);
    I.has_f = false;
    if (f_vertex)
        for (size_t K = 0; K < N; ++K)
            for (int i = 0; i < 3; ++i) {
                fcell[K * 3 + i] = f_vertex[h->hm.cells[3 * K + i]];
                if (fcell[K * 3 + i] != 0.0) I.has_f = true;
            }
    // state buffers: 2 + 2 * kImexMaxStages state vectors (stage state, stage
    // right-hand side, the two rates of every stage)
    I.nq = nq;
    const size_t nbuf = size_t(2 + 2 * kImexMaxStages) * nq;
    cudaError_t e = cudaMalloc(reinterpret_cast<void **>(&I.fcell), sizeof(double) * N * 3);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&I.lam), sizeof(double) * size_t(h->NT));
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&I.lam_out), sizeof(double) * size_t(h->NT));
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&I.buf), sizeof(double) * nbuf);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(I.fcell, fcell.data(), sizeof(double) * N * 3, cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) {
        imex_free(I);
        return imex_fail(h, e == cudaErrorMemoryAllocation ? HDG_ENOMEM : HDG_ECUDA,
                         std::string("hdg_imex_init: ") + cudaGetErrorString(e));
    }
    I.ready = true;
    return HDG_OK;
}

extern "C" int hdg_imex_rates_dev(hdg_handle *h, const double *u, const double *hh, double *nu, double *nh,
                                  double *lu, double *lh) {
    if (!h) return HDG_EINVAL;
    if (!h->imex.ready) return imex_fail(h, HDG_ESTATE, "hdg_imex_init has not run on this handle");
    if (!u || !hh || !lu || !lh || (!nu) != (!nh)) return imex_fail(h, HDG_EINVAL, "NULL pointer argument");
    cudaError_t e = account_launch(h, HDG_PROF_IMEX, 2, [&]() { return launch_imex_rates(h, u, hh, nu, nh, lu, lh); });
    if (e != cudaSuccess) return imex_fail(h, HDG_ECUDA, std::string("hdg_imex_rates_dev: ") + cudaGetErrorString(e));
    return HDG_OK;
}

extern "C" int hdg_imex_step_dev(hdg_handle *h, int scheme, double theta, double dt, double *u, double *hh,
                                 hdg_solve_info *info) {
    if (!h) return HDG_EINVAL;
    Imex &I = h->imex;
    if (!I.ready) return imex_fail(h, HDG_ESTATE, "hdg_imex_init has not run on this handle");
    if (!u || !hh) return imex_fail(h, HDG_EINVAL, "NULL pointer argument");
    if (scheme < HDG_IMEX_THETA || scheme > HDG_IMEX_ARS3) return imex_fail(h, HDG_EINVAL, "unknown IMEX scheme");
    if (!(dt > 0)) return imex_fail(h, HDG_EINVAL, "dt must be positive");
    if (scheme == HDG_IMEX_THETA && !(theta > 0 && theta <= 1))
        return imex_fail(h, HDG_EINVAL, "theta must be in (0, 1]");
    const Tableau T = tableau(scheme, theta);
    // every implicit stage of these schemes has the same a~_ii: one operator
    double alpha = 0.0;
    for (int i = 0; i < T.s; ++i)
        if (T.at[i][i] != 0.0) alpha = T.at[i][i];
    const double tau = alpha * dt;
    if (!h->condensed || std::fabs(h->prm.tau - tau) > 1e-15 * tau) {
        const int rc = hdg_set_tau(h, tau);
        if (rc) return rc;
    }
    const size_t nq = I.nq, nu_ = size_t(h->N) * 2 * h->np;
    double *Q = I.buf, *R = I.buf + nq;
    double *rn[kImexMaxStages], *rl[kImexMaxStages];
    for (int i = 0; i < kImexMaxStages; ++i) {
        rn[i] = I.buf + (2 + 2 * i) * nq;
        rl[i] = I.buf + (3 + 2 * i) * nq;
    }
    cudaStream_t s = h->stream;
    hdg_solve_info acc{};
    int status = HDG_OK;
    const bool expl_f = I.has_f;
    // out = q0 + dt sum_{j < n} (a_j n~_j + at_j l~_j), the terms whose coefficient is zero
    // left out; q0 stays in the caller's u, h until the last combination replaces it
    auto combine = [&](int n, const double *a_, const double *at_, double *ou, double *oh) {
        Combo c;
        for (int j = 0; expl_f && j < n; ++j)
            if (a_[j] != 0.0) {
                c.c[c.k] = a_[j];
                c.x[c.k++] = rn[j];
            }
        c.kn = c.k;
        for (int j = 0; j < n; ++j)
            if (at_[j] != 0.0) {
                c.c[c.k] = at_[j];
                c.x[c.k++] = rl[j];
            }
        return account_launch(h, HDG_PROF_IMEX, 1, [&]() {
            imex_combine_kernel<<<nblocks(nq, 256 * kCombU), 256, 0, s>>>(nu_, nq, u, hh, c, dt, ou, oh);
            return cudaGetLastError();
        });
    };
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < T.s; ++i) {
        // stage right-hand side r_i = q0 + dt sum_{j<i} (a_ij n~_j + a~_ij l~_j)
        const double *Qu, *Qh;
        if (i == 0 && T.at[0][0] == 0.0) {
            Qu = u;                                     // explicit first stage: Q_1 = q0
            Qh = hh;
        } else {
            e = combine(i, T.a[i], T.at[i], R, R + nu_);
            if (e != cudaSuccess) return imex_fail(h, HDG_ECUDA, std::string("imex combine: ") + cudaGetErrorString(e));
            if (T.at[i][i] != 0.0) {
                hdg_solve_info si{};
                int rc = hdg_solve_dev(h, R, R + nu_, I.lam_out, &si);
                acc.iters += si.iters;
                acc.outer += si.outer;
                acc.true_rel_res = std::max(acc.true_rel_res, si.true_rel_res);
                acc.est_rel_res = std::max(acc.est_rel_res, si.est_rel_res);
                if (rc && !status) status = rc;
                if (rc == HDG_ECUDA || rc == HDG_ENAN) break;
                // the stage's recovery from what its step 1 kept (two-float handles), else from R
                const bool kz = solve_kept_z(h);
                rc = hdg_recover_dev(h, kz ? nullptr : R, kz ? nullptr : R + nu_, nullptr, Q, Q + nu_);
                if (rc) return rc;
                Qu = Q;
            } else {
                Qu = R;                                 // M Q = M r: a mass solve in function space
            }
            Qh = Qu + nu_;
        }
        // the stage's rates n~(Q_i), l~(Q_i), those that a later stage or the new state takes
        // (ARS2 never uses the first stage's l~: its weight and its column are zero)
        bool need_n = T.b[i] != 0.0, need_l = T.bt[i] != 0.0;
        for (int j = i + 1; j < T.s; ++j) {
            need_n |= T.a[j][i] != 0.0;
            need_l |= T.at[j][i] != 0.0;
        }
        need_n &= expl_f;
        if (!need_n && !need_l) continue;
        e = account_launch(h, HDG_PROF_IMEX, need_l ? 2 : 1, [&]() {
            return launch_imex_rates(h, Qu, Qh, need_n ? rn[i] : nullptr, nullptr, need_l ? rl[i] : nullptr,
                                     need_l ? rl[i] + nu_ : nullptr);
        });
        if (e != cudaSuccess) return imex_fail(h, HDG_ECUDA, std::string("imex rates: ") + cudaGetErrorString(e));
    }
    if (status == HDG_ECUDA || status == HDG_ENAN) {
        acc.status = status;
        if (info) *info = acc;
        return status;
    }
    // q1 = q0 + dt sum_i (b_i n~_i + b~_i l~_i), written into the caller's u, h
    e = combine(T.s, T.b, T.bt, u, hh);
    if (e != cudaSuccess) return imex_fail(h, HDG_ECUDA, std::string("hdg_imex_step_dev: ") + cudaGetErrorString(e));
    acc.status = status;
    if (info) *info = acc;
    return status;
}
