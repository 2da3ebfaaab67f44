// Trace-space kernels: the facet-row trace operator and everything that lives
// on the facets.
//
// Internal trace vectors are stored node-major, x[r * NF + e] (node r of facet
// e), so that every thread (one facet) reads and writes coalesced planes.  The
// caller-facing lambda layout [NF][p+1] is converted at the API boundary.
//
// Trace operator (Eq. schur_system): one thread per facet e computes its p+1
// rows  y_{e,r} = sum_{b<5} sum_c Sval[(r*5+b)*PP+c][e] x_{src(b),c}  with
// src(0) = e and src(b) = nbr[b-1][e]: the diagonal block (both cells' S_K
// summed) and the four blocks that couple e to the other two facets of each of
// its cells.  The block-Jacobi smoother (the smoother of Alg. twolevel_vcycle,
// with the facet blocks inverted exactly) is the same pass followed by
//   x_new = x + omega D_e^-1 (b - S x)  on the facet's p+1 values.
#include "common.h"

#include <cuda_bf16.h>
#include <type_traits>

namespace hdg {

// launch family of this file for pdl_launch (facet-row kernels)
constexpr unsigned kPdlFamily = 1;

namespace {

template <typename TO> __device__ __forceinline__ TO convert_to(double v);
template <> __device__ __forceinline__ double convert_to<double>(double v) { return v; }
template <> __device__ __forceinline__ float convert_to<float>(double v) { return to_float(v); }

// Operator values are packed in 16-byte groups: element j of facet e lives at
// group (j / G, e), lane j % G, with G = 16 / sizeof(storage); every thread
// issues one 16-byte load per group.  Storage FP64 (G = 2), FP32 (G = 4) or
// BF16 (G = 8, unpacked to FP32); arithmetic in the compute type T.
template <typename ST> struct Pack;
template <> struct Pack<double> {
    static constexpr int G = 2;
    using V = double2;
    __device__ static void unpack(const V &v, double (&o)[2]) { o[0] = v.x; o[1] = v.y; }
};
template <> struct Pack<float> {
    static constexpr int G = 4;
    using V = float4;
    __device__ static void unpack(const V &v, float (&o)[4]) { o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w; }
};
template <> struct Pack<__nv_bfloat16> {
    static constexpr int G = 8;
    using V = uint4;
    __device__ static void unpack(const V &v, float (&o)[8]) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            o[2 * k] = __uint_as_float(w[k] << 16);
            o[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
        }
    }
};
template <typename ST> using unpacked_t = typename std::conditional<std::is_same<ST, double>::value, double, float>::type;

// gather the p+1 trace values of the facet and its four neighbours
template <int P, typename T>
__device__ __forceinline__ void gather_x(const int32_t *__restrict__ nbr, const T *__restrict__ x, int e, size_t NF,
                                         T (&xs)[5][P + 1]) {
    int src[5];
    src[0] = e;
#pragma unroll
    for (int b = 1; b < 5; ++b) src[b] = __ldg(nbr + size_t(b - 1) * NF + e);
#pragma unroll
    for (int b = 0; b < 5; ++b)
#pragma unroll
        for (int c = 0; c < P + 1; ++c) xs[b][c] = x[size_t(c) * NF + src[b]];
}

// y_r = sum_{b,c} S[(r*5+b)*PP+c] xs[b][c] with packed loads
template <int P, typename T, typename ST>
__device__ __forceinline__ void facet_rows_packed(const ST *__restrict__ Sval, int e, size_t NF,
                                                  const T (&xs)[5][P + 1], T (&y)[P + 1]) {
    constexpr int PP = P + 1, NS = 5 * PP * PP, G = Pack<ST>::G, NQ = (NS + G - 1) / G;
    using V = typename Pack<ST>::V;
    const V *Sp = reinterpret_cast<const V *>(Sval);
#pragma unroll
    for (int r = 0; r < PP; ++r) y[r] = T(0);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const V v = __ldg(Sp + size_t(q) * NF + e);
        unpacked_t<ST> o[G];
        Pack<ST>::unpack(v, o);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int j = q * G + g;
            if (j < NS) {
                const int r = j / (5 * PP), rem = j % (5 * PP), b = rem / PP, c = rem % PP;
                y[r] = fma(T(o[g]), xs[b][c], y[r]);
            }
        }
    }
}

// y_r = sum over the four neighbour blocks of H[(r*4+b)*PP+c] xs[1+b][c] with packed loads
template <int P, typename T, typename ST>
__device__ __forceinline__ void hat_rows_packed(const ST *__restrict__ H, int e, size_t NF, const T (&xs)[5][P + 1],
                                                T (&y)[P + 1]) {
    constexpr int PP = P + 1, NS = 4 * PP * PP, G = Pack<ST>::G, NQ = (NS + G - 1) / G;
    using V = typename Pack<ST>::V;
    const V *Hp = reinterpret_cast<const V *>(H);
#pragma unroll
    for (int r = 0; r < PP; ++r) y[r] = T(0);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const V v = __ldg(Hp + size_t(q) * NF + e);
        unpacked_t<ST> o[G];
        Pack<ST>::unpack(v, o);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int j = q * G + g;
            if (j < NS) {
                const int r = j / (4 * PP), rem = j % (4 * PP), b = rem / PP, c = rem % PP;
                y[r] = fma(T(o[g]), xs[1 + b][c], y[r]);
            }
        }
    }
}

// out_r = sum_c Dinv[r*PP+c] v_c with packed loads
template <int P, typename T, typename DT>
__device__ __forceinline__ void block_solve_packed(const DT *__restrict__ Dinv, int e, size_t NF, const T (&v)[P + 1],
                                                   T (&out)[P + 1]) {
    constexpr int PP = P + 1, ND = PP * PP, G = Pack<DT>::G, NQ = (ND + G - 1) / G;
    using V = typename Pack<DT>::V;
    const V *Dp = reinterpret_cast<const V *>(Dinv);
#pragma unroll
    for (int r = 0; r < PP; ++r) out[r] = T(0);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const V w = __ldg(Dp + size_t(q) * NF + e);
        unpacked_t<DT> o[G];
        Pack<DT>::unpack(w, o);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int j = q * G + g;
            if (j < ND) out[j / PP] = fma(T(o[g]), v[j % PP], out[j / PP]);
        }
    }
}

// FP32 facet-row kernels are bound by memory latency: cap registers so six
// 256-thread blocks fit per SM (one wave over the facets of large meshes);
// FP64 ones are bound by the FP64 pipe and keep their registers.
template <typename T> struct MinBlocks { static constexpr int value = sizeof(T) == 4 ? 6 : 1; };
template <int P, typename T, typename ST>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) apply_kernel(int NF, const ST *__restrict__ Sval, const int32_t *__restrict__ nbr,
                                                    const T *__restrict__ x, T *__restrict__ y) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    T xs[5][P + 1], v[P + 1];
    gather_x<P, T>(nbr, x, e, NF, xs);
    facet_rows_packed<P, T, ST>(Sval, e, NF, xs, v);
#pragma unroll
    for (int r = 0; r <= P; ++r) y[size_t(r) * NF + e] = v[r];
}

// y = S x (as apply_kernel) and h = V^T y over the first k basis vectors (the
// first Gram-Schmidt pass of an Arnoldi step): each block sums its facets'
// rows, G vectors at a time, into per-block partials; the last block to
// finish adds the partials in block order (deterministic) into h, and writes -h
// rounded to the vector type to hneg (the coefficients of the update that follows).
// The sums over a warp by halving exchanges (warp_sums) and the warps' sums for all
// vectors after one barrier: 63.1 instead of 70.4 us on 196,608 facets at p = 3 in FP64
// (bound by the FP64 pipe: 80 + 4 k FMAs per facet, and k adds per block by the last one),
// 9.6 instead of 11.5 us on 768 facets (latency).  In FP32 what bounds it is the latency
// of the loads: B blocks per SM (launch_apply_dots_t) decide how many a thread
// has in flight.
template <int P, typename T, typename ST, int B>
__device__ __forceinline__ void apply_dots_kernel_impl(int bid_, int nb_, int NF, const ST *__restrict__ Sval,
                                                       const int32_t *__restrict__ nbr, const T *__restrict__ x,
                                                       T *__restrict__ y, const T *__restrict__ V, size_t ld, int k,
                                                       double *__restrict__ partial,
                                                       unsigned int *__restrict__ counter, double *__restrict__ h,
                                                       T *__restrict__ hneg) {
    using A = typename std::conditional<std::is_same<T, double>::value, double, float>::type;
    constexpr int PP = P + 1, G = sizeof(T) == 8 ? 8 : B > 4 ? 4 : 8, KM = 72;   // (FP32, B = 6: 40 registers)
    __shared__ A red[8][KM];                   // the warps' sums of every vector (k <= 65)
    __shared__ bool last;
    const int e = bid_ * blockDim.x + threadIdx.x;
    const bool valid = e < NF;
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, nwarp = blockDim.x / 32;
    T v[PP];
    if (valid) {
        T xs[5][PP];
        gather_x<P, T>(nbr, x, e, NF, xs);
        facet_rows_packed<P, T, ST>(Sval, e, NF, xs, v);
#pragma unroll
        for (int r = 0; r < PP; ++r) y[size_t(r) * NF + e] = v[r];
    } else {
#pragma unroll
        for (int r = 0; r < PP; ++r) v[r] = T(0);
    }
    for (int i0 = 0; i0 < k; i0 += G) {
        A acc[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            A a = A(0);
            if (valid && i0 + g < k) {
#pragma unroll
                for (int r = 0; r < PP; ++r) a = fma(A(V[size_t(i0 + g) * ld + size_t(r) * NF + e]), A(v[r]), a);
            }
            acc[g] = a;
        }
        int which;
        const A t = warp_sums<G>(acc, which);
        if (lane % (32 / G) == 0) red[warp][i0 + which] = t;
    }
    __syncthreads();
    // eight lanes per vector add the warps' sums (whole warps take part)
    for (int i0 = 0; i0 < k; i0 += int(blockDim.x) / 8) {
        const int i = i0 + int(threadIdx.x) / 8, q = threadIdx.x % 8;
        A t = (i < k && q < nwarp) ? red[q][i] : A(0);
#pragma unroll
        for (int off = 4; off > 0; off /= 2) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (i < k && q == 0) {
            partial[size_t(i) * nb_ + bid_] = double(t);
            __threadfence();                   // the partial is visible before the count
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(counter, 1u) == nb_ - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    finish_partials(partial, int(nb_), k, h);
    if (hneg)
        for (int i = threadIdx.x; i < k; i += blockDim.x) hneg[i] = T(-h[i]);
    if (threadIdx.x == 0) *counter = 0u;
}
template <int P, typename T, typename ST, int B>
__global__ void __launch_bounds__(256, B) apply_dots_kernel(int NF, const ST *__restrict__ Sval,
                                                            const int32_t *__restrict__ nbr, const T *__restrict__ x,
                                                            T *__restrict__ y, const T *__restrict__ V, size_t ld,
                                                            int k, double *__restrict__ partial,
                                                            unsigned int *__restrict__ counter,
                                                            double *__restrict__ h, T *__restrict__ hneg) {
    pdl_wait();
    apply_dots_kernel_impl<P, T, ST, B>(blockIdx.x, gridDim.x, NF, Sval, nbr, x, y, V, ld, k, partial, counter, h, hneg);
}
template <int P, typename T, typename ST, int B>
struct apply_dots_kernel_args {
    int nb_;
    int NF;
    const ST *Sval;
    const int32_t *nbr;
    const T *x;
    T *y;
    const T *V;
    size_t ld;
    int k;
    double *partial;
    unsigned int *counter;
    double *h;
    T *hneg;
};
template <int P, typename T, typename ST, int B>
__global__ void __launch_bounds__(256, B) apply_dots_kernel_multi(const __grid_constant__ MultiP<apply_dots_kernel_args<P, T, ST, B>> M) {
    pdl_wait();
    int b_;
    const apply_dots_kernel_args<P, T, ST, B> &q_ = M.a[merge_find(M.start, M.n, b_)];
    apply_dots_kernel_impl<P, T, ST, B>(b_, q_.nb_, q_.NF, q_.Sval, q_.nbr, q_.x, q_.y, q_.V, q_.ld, q_.k, q_.partial,
        q_.counter, q_.h, q_.hneg);
}
template <int P, typename T, typename ST, int B>
void apply_dots_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int NF, const ST *Sval,
                          const int32_t *nbr, const T *x, T *y, const T *V, size_t ld, int k, double *partial,
                          unsigned int *counter, double *h, T *hneg) {
    if (Recorder *r_ = batch_recorder()) {
        apply_dots_kernel_args<P, T, ST, B> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.NF = NF;
        q_.Sval = Sval;
        q_.nbr = nbr;
        q_.x = x;
        q_.y = y;
        q_.V = V;
        q_.ld = ld;
        q_.k = k;
        q_.partial = partial;
        q_.counter = counter;
        q_.h = h;
        q_.hneg = hneg;
        batch_record(r_, reinterpret_cast<const void *>(&apply_dots_kernel_multi<P, T, ST, B>), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &apply_dots_kernel<P, T, ST, B>, grid_, block_, smem_, s_, NF, Sval, nbr, x, y, V, ld, k, partial, counter, h, hneg);
}


template <int P, typename T, typename ST>
__device__ __forceinline__ void residual_kernel_impl(int bid_, int nb_, int NF, const ST *__restrict__ Sval,
                                                     const int32_t *__restrict__ nbr, const T *__restrict__ b,
                                                     const T *__restrict__ x, T *__restrict__ res) {
    const int e = bid_ * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    T xs[5][P + 1], v[P + 1];
    gather_x<P, T>(nbr, x, e, NF, xs);
    facet_rows_packed<P, T, ST>(Sval, e, NF, xs, v);
#pragma unroll
    for (int r = 0; r <= P; ++r) res[size_t(r) * NF + e] = b[size_t(r) * NF + e] - v[r];
}
template <int P, typename T, typename ST>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) residual_kernel(int NF, const ST *__restrict__ Sval,
                                                                            const int32_t *__restrict__ nbr,
                                                                            const T *__restrict__ b,
                                                                            const T *__restrict__ x,
                                                                            T *__restrict__ res) {
    pdl_wait();
    residual_kernel_impl<P, T, ST>(blockIdx.x, gridDim.x, NF, Sval, nbr, b, x, res);
}
template <int P, typename T, typename ST>
struct residual_kernel_args {
    int nb_;
    int NF;
    const ST *Sval;
    const int32_t *nbr;
    const T *b;
    const T *x;
    T *res;
};
template <int P, typename T, typename ST>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) residual_kernel_multi(const __grid_constant__ MultiP<residual_kernel_args<P, T, ST>> M) {
    pdl_wait();
    int b_;
    const residual_kernel_args<P, T, ST> &q_ = M.a[merge_find(M.start, M.n, b_)];
    residual_kernel_impl<P, T, ST>(b_, q_.nb_, q_.NF, q_.Sval, q_.nbr, q_.b, q_.x, q_.res);
}
template <int P, typename T, typename ST>
void residual_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int NF, const ST *Sval,
                        const int32_t *nbr, const T *b, const T *x, T *res) {
    if (Recorder *r_ = batch_recorder()) {
        residual_kernel_args<P, T, ST> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.NF = NF;
        q_.Sval = Sval;
        q_.nbr = nbr;
        q_.b = b;
        q_.x = x;
        q_.res = res;
        batch_record(r_, reinterpret_cast<const void *>(&residual_kernel_multi<P, T, ST>), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &residual_kernel<P, T, ST>, grid_, block_, smem_, s_, NF, Sval, nbr, b, x, res);
}


// The smoothing sweeps, on one of two sets of operators.  With HAT, on the rows of D^-1 S:
// with b standing for bh = D^-1 b (formed once per preconditioner application by the first
// sweep), op for H, the four neighbour blocks of D^-1 S (the diagonal block is the identity),
//   D_e^-1 (b - S x)_e = bh_e - x_e - sum_b H_b x_nbr(b),
// so a sweep reads 4 (p+1)^2 operator values per facet instead of 6 (p+1)^2 (S and the
// inverse block).  Without, op is S, blk the inverse block: kept for FP32 handles of the
// sizes where S, which the Krylov space applies too, stays in L2 from one kernel to the
// next (hat_pays32 in api.cu).  What bounds a sweep is the operator's stream (HBM and L2);
// in FP64 the FP64 pipe, 64 instead of 96 FMAs per facet at p = 3: the step with 196,608
// facets takes 3440 instead of 3650 us in FP64, the one with 491,520 (p = 2, FP32) 2435
// instead of 2683, with 30,000 (p = 4, BF16) 1175 instead of 1258.
//
// The residual before the coarse correction, res = b - S x (with HAT as D (D^-1 (b - S x)),
// blk the diagonal block D), and the part of the first post-smoothing sweep that does not
// wait for the correction, y = x + omega D^-1 (b - S x).
template <int P, typename T, typename ST, bool HAT>
__device__ __forceinline__ void residual_smooth_kernel_impl(int bid_, int nb_, int NF, const ST *__restrict__ op,
                                                            const T *__restrict__ blk,
                                                            const int32_t *__restrict__ nbr, const T *__restrict__ b,
                                                            const T *__restrict__ x, T *__restrict__ res,
                                                            T *__restrict__ y, T omega) {
    const int e = bid_ * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    T xs[5][P + 1], v[P + 1], d[P + 1];
    gather_x<P, T>(nbr, x, e, NF, xs);
    if constexpr (HAT) hat_rows_packed<P, T, ST>(op, e, NF, xs, v);
    else facet_rows_packed<P, T, ST>(op, e, NF, xs, v);
#pragma unroll
    for (int r = 0; r <= P; ++r) {
        if constexpr (HAT) v[r] = (b[size_t(r) * NF + e] - xs[0][r]) - v[r];
        else v[r] = b[size_t(r) * NF + e] - v[r];
        (HAT ? y : res)[size_t(r) * NF + e] = HAT ? fma(omega, v[r], xs[0][r]) : v[r];
    }
    block_solve_packed<P, T, T>(blk, e, NF, v, d);
#pragma unroll
    for (int r = 0; r <= P; ++r) (HAT ? res : y)[size_t(r) * NF + e] = HAT ? d[r] : fma(omega, d[r], xs[0][r]);
}
template <int P, typename T, typename ST, bool HAT>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) residual_smooth_kernel(int NF, const ST *__restrict__ op,
                                                                                   const T *__restrict__ blk,
                                                                                   const int32_t *__restrict__ nbr,
                                                                                   const T *__restrict__ b,
                                                                                   const T *__restrict__ x,
                                                                                   T *__restrict__ res,
                                                                                   T *__restrict__ y, T omega) {
    pdl_wait();
    residual_smooth_kernel_impl<P, T, ST, HAT>(blockIdx.x, gridDim.x, NF, op, blk, nbr, b, x, res, y, omega);
}
template <int P, typename T, typename ST, bool HAT>
struct residual_smooth_kernel_args {
    int nb_;
    int NF;
    const ST *op;
    const T *blk;
    const int32_t *nbr;
    const T *b;
    const T *x;
    T *res;
    T *y;
    T omega;
};
template <int P, typename T, typename ST, bool HAT>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) residual_smooth_kernel_multi(const __grid_constant__ MultiP<residual_smooth_kernel_args<P, T, ST, HAT>> M) {
    pdl_wait();
    int b_;
    const residual_smooth_kernel_args<P, T, ST, HAT> &q_ = M.a[merge_find(M.start, M.n, b_)];
    residual_smooth_kernel_impl<P, T, ST, HAT>(b_, q_.nb_, q_.NF, q_.op, q_.blk, q_.nbr, q_.b, q_.x, q_.res, q_.y,
        q_.omega);
}
template <int P, typename T, typename ST, bool HAT>
void residual_smooth_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int NF, const ST *op,
                               const T *blk, const int32_t *nbr, const T *b, const T *x, T *res, T *y, T omega) {
    if (Recorder *r_ = batch_recorder()) {
        residual_smooth_kernel_args<P, T, ST, HAT> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.NF = NF;
        q_.op = op;
        q_.blk = blk;
        q_.nbr = nbr;
        q_.b = b;
        q_.x = x;
        q_.res = res;
        q_.y = y;
        q_.omega = omega;
        batch_record(r_, reinterpret_cast<const void *>(&residual_smooth_kernel_multi<P, T, ST, HAT>), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &residual_smooth_kernel<P, T, ST, HAT>, grid_, block_, smem_, s_, NF, op, blk, nbr, b, x, res, y, omega);
}


// One sweep x_out = x + omega D_e^-1 (b - S x)_e; with CHEB, a step of the
// Chebyshev iteration x_out = x + omega D_e^-1 (b - S x)_e + beta (x - x_prev)
// (x_prev null: the previous iterate is zero).  x_out may alias x_prev: each
// thread reads x_prev only at its own facet before writing it.
template <int P, typename T, typename ST, bool HAT, bool CHEB>
__device__ __forceinline__ void smooth_kernel_impl(int bid_, int nb_, int NF, const ST *__restrict__ op, const T *__restrict__ blk,
                                                   const int32_t *__restrict__ nbr, const T *__restrict__ b,
                                                   const T *__restrict__ x, T *xout, T omega, T beta,
                                                   const T *xprev) {
    constexpr int PP = P + 1;
    const int e = bid_ * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    T xs[5][PP], v[PP], d[PP];
    gather_x<P, T>(nbr, x, e, NF, xs);
    if constexpr (HAT) {
        hat_rows_packed<P, T, ST>(op, e, NF, xs, v);
#pragma unroll
        for (int r = 0; r < PP; ++r) d[r] = (b[size_t(r) * NF + e] - xs[0][r]) - v[r];
    } else {
        facet_rows_packed<P, T, ST>(op, e, NF, xs, v);
#pragma unroll
        for (int r = 0; r < PP; ++r) v[r] = b[size_t(r) * NF + e] - v[r];
        block_solve_packed<P, T, T>(blk, e, NF, v, d);
    }
#pragma unroll
    for (int r = 0; r < PP; ++r) {
        T o = fma(omega, d[r], xs[0][r]);
        if constexpr (CHEB) {
            const T xp = xprev ? xprev[size_t(r) * NF + e] : T(0);
            o = fma(beta, xs[0][r] - xp, o);
        }
        xout[size_t(r) * NF + e] = o;
    }
}
template <int P, typename T, typename ST, bool HAT, bool CHEB>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) smooth_kernel(int NF, const ST *__restrict__ op, const T *__restrict__ blk,
                                                                          const int32_t *__restrict__ nbr,
                                                                          const T *__restrict__ b,
                                                                          const T *__restrict__ x, T *xout, T omega,
                                                                          T beta, const T *xprev) {
    pdl_wait();
    smooth_kernel_impl<P, T, ST, HAT, CHEB>(blockIdx.x, gridDim.x, NF, op, blk, nbr, b, x, xout, omega, beta, xprev);
}
template <int P, typename T, typename ST, bool HAT, bool CHEB>
struct smooth_kernel_args {
    int nb_;
    int NF;
    const ST *op;
    const T *blk;
    const int32_t *nbr;
    const T *b;
    const T *x;
    T *xout;
    T omega;
    T beta;
    const T *xprev;
};
template <int P, typename T, typename ST, bool HAT, bool CHEB>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) smooth_kernel_multi(const __grid_constant__ MultiP<smooth_kernel_args<P, T, ST, HAT, CHEB>> M) {
    pdl_wait();
    int b_;
    const smooth_kernel_args<P, T, ST, HAT, CHEB> &q_ = M.a[merge_find(M.start, M.n, b_)];
    smooth_kernel_impl<P, T, ST, HAT, CHEB>(b_, q_.nb_, q_.NF, q_.op, q_.blk, q_.nbr, q_.b, q_.x, q_.xout, q_.omega,
        q_.beta, q_.xprev);
}
template <int P, typename T, typename ST, bool HAT, bool CHEB>
void smooth_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int NF, const ST *op, const T *blk,
                      const int32_t *nbr, const T *b, const T *x, T *xout, T omega, T beta,
                      const T *xprev) {
    if (Recorder *r_ = batch_recorder()) {
        smooth_kernel_args<P, T, ST, HAT, CHEB> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.NF = NF;
        q_.op = op;
        q_.blk = blk;
        q_.nbr = nbr;
        q_.b = b;
        q_.x = x;
        q_.xout = xout;
        q_.omega = omega;
        q_.beta = beta;
        q_.xprev = xprev;
        batch_record(r_, reinterpret_cast<const void *>(&smooth_kernel_multi<P, T, ST, HAT, CHEB>), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &smooth_kernel<P, T, ST, HAT, CHEB>, grid_, block_, smem_, s_, NF, op, blk, nbr, b, x, xout, omega, beta, xprev);
}


// First post-smoothing sweep with the coarse correction folded in: from x' = x + pi e_c,
// x_out = x' + omega D_e^-1 (b - S x')_e.  The residual before the correction was formed
// for the restriction, with y = x + omega D^-1 (b - S x) (residual_smooth_kernel), and the
// rows of S pi couple a facet to four vertices only, its own two and the two opposite it in
// its cells: with Q = D^-1 S pi stored ([row][facet], one 4-vector each),
//   x_out = y + pi e_c - omega Q_e (e_c at the four vertices),
// so the sweep reads 4 (p+1) operator entries per facet instead of 6 (p+1)^2 and gathers
// four vertex values instead of five facets' traces and ten vertices.  Bound by HBM and L2
// latency: 9.1 instead of 28.4 us on 491,520 facets (p = 2, FP32), 16.0 instead of 60.1 us
// on 196,608 (p = 3, FP64, where the old form was bound by the FP64 pipe); the residual
// kernel takes 2.7 and 7 us more for y.  On the 196,608-facet p = 3 FP32 solve, whose
// operator nearly fits L2, the step time stays (6.3 + 15 us for the two post-smoothing
// sweeps instead of 13.4 + 10.5: the second now brings the operator from HBM itself).
// With X0, x' on the facet itself is also stored to x0out (the previous iterate of the
// Chebyshev step that follows).  xout may alias y.
template <typename T> struct Vec4;
template <> struct Vec4<float> {
    using type = float4;
};
template <> struct Vec4<double> {
    struct __align__(16) type { double x, y, z, w; };
};
template <int P, typename T, bool X0 = false>
__device__ __forceinline__ void smooth_prolong_kernel_impl(int bid_, int nb_, int NF, const T *__restrict__ Q,
                                                           const int32_t *__restrict__ fverts,
                                                           const int32_t *__restrict__ fopp,
                                                           const T *__restrict__ ec, const T *y,
                                                           const T *__restrict__ x, T *xout, T omega,
                                                           T *__restrict__ x0out) {
    using V = typename Vec4<T>::type;
    constexpr int PP = P + 1;
    const int e = bid_ * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    const int2 lv = __ldg(reinterpret_cast<const int2 *>(fverts) + e), ov = __ldg(reinterpret_cast<const int2 *>(fopp) + e);
    V q[PP];
#pragma unroll
    for (int r = 0; r < PP; ++r) q[r] = reinterpret_cast<const V *>(Q)[size_t(r) * NF + e];
    const T lo = ec[lv.x], hi = ec[lv.y], oa = ec[ov.x], ob = ec[ov.y];
#pragma unroll
    for (int r = 0; r < PP; ++r) {
        const T qc = fma(q[r].x, lo, fma(q[r].y, hi, fma(q[r].z, oa, q[r].w * ob)));
        const T t = T(r) / T(P), pc = fma(T(1) - t, lo, t * hi);
        if constexpr (X0) x0out[size_t(r) * NF + e] = x[size_t(r) * NF + e] + pc;
        xout[size_t(r) * NF + e] = fma(-omega, qc, y[size_t(r) * NF + e] + pc);
    }
}
template <int P, typename T, bool X0 = false>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) smooth_prolong_kernel(int NF, const T *__restrict__ Q,
                                                                                  const int32_t *__restrict__ fverts,
                                                                                  const int32_t *__restrict__ fopp,
                                                                                  const T *__restrict__ ec, const T *y,
                                                                                  const T *__restrict__ x, T *xout,
                                                                                  T omega, T *__restrict__ x0out) {
    pdl_wait();
    smooth_prolong_kernel_impl<P, T, X0>(blockIdx.x, gridDim.x, NF, Q, fverts, fopp, ec, y, x, xout, omega, x0out);
}
template <int P, typename T, bool X0 = false>
struct smooth_prolong_kernel_args {
    int nb_;
    int NF;
    const T *Q;
    const int32_t *fverts;
    const int32_t *fopp;
    const T *ec;
    const T *y;
    const T *x;
    T *xout;
    T omega;
    T *x0out;
};
template <int P, typename T, bool X0 = false>
__global__ void __launch_bounds__(256, MinBlocks<T>::value) smooth_prolong_kernel_multi(const __grid_constant__ MultiP<smooth_prolong_kernel_args<P, T, X0>> M) {
    pdl_wait();
    int b_;
    const smooth_prolong_kernel_args<P, T, X0> &q_ = M.a[merge_find(M.start, M.n, b_)];
    smooth_prolong_kernel_impl<P, T, X0>(b_, q_.nb_, q_.NF, q_.Q, q_.fverts, q_.fopp, q_.ec, q_.y, q_.x, q_.xout,
        q_.omega, q_.x0out);
}
template <int P, typename T, bool X0 = false>
void smooth_prolong_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int NF, const T *Q,
                              const int32_t *fverts, const int32_t *fopp, const T *ec, const T *y, const T *x, T *xout,
                              T omega, T *x0out) {
    if (Recorder *r_ = batch_recorder()) {
        smooth_prolong_kernel_args<P, T, X0> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.NF = NF;
        q_.Q = Q;
        q_.fverts = fverts;
        q_.fopp = fopp;
        q_.ec = ec;
        q_.y = y;
        q_.x = x;
        q_.xout = xout;
        q_.omega = omega;
        q_.x0out = x0out;
        batch_record(r_, reinterpret_cast<const void *>(&smooth_prolong_kernel_multi<P, T, X0>), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &smooth_prolong_kernel<P, T, X0>, grid_, block_, smem_, s_, NF, Q, fverts, fopp, ec, y, x, xout, omega,
        x0out);
}

// The smoother's operators from the packed FP64 operator, once per condensation, in FP64
// and rounded once for the FP32 and BF16 copies: H, the four neighbour blocks of D^-1 S
// (element (r*4+b)*PP+c, packed), the diagonal block D (packed), and, with PROL, Q = D^-1 S
// pi: row r of facet e against the facet's own vertices and the two opposite it.  A
// neighbour facet of cell s joins two of that cell's three vertices; its row's entries are
// summed with weights 1 - t_c and t_c onto its lower and higher vertex.
struct HatOut {
    double *H, *D, *Q;
    float *H32, *D32, *Q32;
    __nv_bfloat16 *H16;
};
template <int P, bool PROL>
__global__ void hat_op_kernel(int NF, const double *__restrict__ Sval, const double *__restrict__ Dinv,
                              const int32_t *__restrict__ nbr, const int32_t *__restrict__ fverts, HatOut o) {
    constexpr int PP = P + 1;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    double d[PP][PP], w[PP][4];
#pragma unroll
    for (int r = 0; r < PP; ++r)
#pragma unroll
        for (int c = 0; c < PP; ++c) {
            d[r][c] = Dinv[packed_index(size_t(r * PP + c), size_t(e), size_t(NF), 2)];
            const double s = Sval[packed_index(size_t(r * 5 * PP + c), size_t(e), size_t(NF), 2)];
            if (o.D) o.D[packed_index(size_t(r * PP + c), size_t(e), size_t(NF), 2)] = s;
            if (o.D32) o.D32[packed_index(size_t(r * PP + c), size_t(e), size_t(NF), 4)] = to_float(s);
        }
    int lo = 0, hi = 0;
    if constexpr (PROL) {
        lo = fverts[2 * e];
        hi = fverts[2 * e + 1];
        // the facet's own block (the identity)
#pragma unroll
        for (int r = 0; r < PP; ++r) {
            w[r][1] = double(r) / double(P);
            w[r][0] = 1.0 - w[r][1];
            w[r][2] = w[r][3] = 0.0;
        }
    }
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
        int s0 = 0, s1 = 0;                    // slots of the neighbour's vertices: 0 lo, 1 hi, 2 / 3 opposite in cell 0 / 1
        if constexpr (PROL) {
            const int f = nbr[size_t(b) * NF + e], v0 = fverts[2 * f], v1 = fverts[2 * f + 1], op = b < 2 ? 2 : 3;
            s0 = v0 == lo ? 0 : v0 == hi ? 1 : op;
            s1 = v1 == lo ? 0 : v1 == hi ? 1 : op;
        }
        double tot[PP], up[PP];
#pragma unroll
        for (int r = 0; r < PP; ++r) tot[r] = up[r] = 0.0;
#pragma unroll
        for (int c = 0; c < PP; ++c) {
            double s[PP];
#pragma unroll
            for (int q = 0; q < PP; ++q)
                s[q] = Sval[packed_index(size_t((q * 5 + 1 + b) * PP + c), size_t(e), size_t(NF), 2)];
#pragma unroll
            for (int r = 0; r < PP; ++r) {
                double v = 0.0;
#pragma unroll
                for (int q = 0; q < PP; ++q) v = fma(d[r][q], s[q], v);
                const size_t j = size_t((r * 4 + b) * PP + c);
                if (o.H) o.H[packed_index(j, size_t(e), size_t(NF), 2)] = v;
                if (o.H32) o.H32[packed_index(j, size_t(e), size_t(NF), 4)] = to_float(v);
                if (o.H16) o.H16[packed_index(j, size_t(e), size_t(NF), 8)] = __double2bfloat16(v);
                if constexpr (PROL) {
                    tot[r] += v;
                    if (c > 0) up[r] = c < P ? fma(v, double(c) / double(P), up[r]) : up[r] + v;
                }
            }
        }
        if constexpr (PROL) {
#pragma unroll
            for (int r = 0; r < PP; ++r)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (s0 == q) w[r][q] += tot[r] - up[r];
                    if (s1 == q) w[r][q] += up[r];
                }
        }
    }
    if constexpr (PROL) {
#pragma unroll
        for (int r = 0; r < PP; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                o.Q[(size_t(r) * NF + e) * 4 + q] = w[r][q];
                if (o.Q32) o.Q32[(size_t(r) * NF + e) * 4 + q] = to_float(w[r][q]);
            }
    }
    // (padding lanes of the last groups are never multiplied)
}


// first sweep from a zero initial guess: bh = D^-1 b (kept for the sweeps that follow;
// null: not wanted), x = omega bh
template <int P, typename T>
__device__ __forceinline__ void smooth_first_kernel_impl(int bid_, int nb_, int NF, const T *__restrict__ Dinv,
                                                         const T *__restrict__ b, T *__restrict__ xout, T *__restrict__ bh, T omega,
                                                         const T *__restrict__ w, const double *__restrict__ hnext,
                                                         T *__restrict__ bout) {
    // with w: the right-hand side is the next Arnoldi vector b = w / h_{j+1,j}
    // (the last Gram-Schmidt step of the previous iteration), also stored to
    // bout; the FP64 reciprocal is formed once per block
    __shared__ double inv_h;
    if (w != nullptr) {
        if (threadIdx.x == 0) inv_h = 1.0 / hnext[0];
        __syncthreads();
    }
    constexpr int PP = P + 1;
    const int e = bid_ * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    T v[PP], d[PP];
    if (w != nullptr) {
        const T inv = T(inv_h);
#pragma unroll
        for (int c = 0; c < PP; ++c) {
            v[c] = w[size_t(c) * NF + e] * inv;
            bout[size_t(c) * NF + e] = v[c];
        }
    } else {
#pragma unroll
        for (int c = 0; c < PP; ++c) v[c] = b[size_t(c) * NF + e];
    }
    block_solve_packed<P, T, T>(Dinv, e, NF, v, d);
#pragma unroll
    for (int r = 0; r < PP; ++r) {
        if (bh) bh[size_t(r) * NF + e] = d[r];
        xout[size_t(r) * NF + e] = omega * d[r];
    }
}
template <int P, typename T>
__global__ void smooth_first_kernel(int NF, const T *__restrict__ Dinv, const T *__restrict__ b, T *__restrict__ xout, T *__restrict__ bh,
                                    T omega, const T *__restrict__ w, const double *__restrict__ hnext,
                                    T *__restrict__ bout) {
    pdl_wait();
    smooth_first_kernel_impl<P, T>(blockIdx.x, gridDim.x, NF, Dinv, b, xout, bh, omega, w, hnext, bout);
}
template <int P, typename T>
struct smooth_first_kernel_args {
    int nb_;
    int NF;
    const T *Dinv;
    const T *b;
    T *xout;
    T *bh;
    T omega;
    const T *w;
    const double *hnext;
    T *bout;
};
template <int P, typename T>
__global__ void smooth_first_kernel_multi(const __grid_constant__ MultiP<smooth_first_kernel_args<P, T>> M) {
    pdl_wait();
    int b_;
    const smooth_first_kernel_args<P, T> &q_ = M.a[merge_find(M.start, M.n, b_)];
    smooth_first_kernel_impl<P, T>(b_, q_.nb_, q_.NF, q_.Dinv, q_.b, q_.xout, q_.bh, q_.omega, q_.w, q_.hnext, q_.bout);
}
template <int P, typename T>
void smooth_first_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int NF, const T *Dinv,
                            const T *b, T *xout, T *bh, T omega, const T *w, const double *hnext, T *bout) {
    if (Recorder *r_ = batch_recorder()) {
        smooth_first_kernel_args<P, T> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.NF = NF;
        q_.Dinv = Dinv;
        q_.b = b;
        q_.xout = xout;
        q_.bh = bh;
        q_.omega = omega;
        q_.w = w;
        q_.hnext = hnext;
        q_.bout = bout;
        batch_record(r_, reinterpret_cast<const void *>(&smooth_first_kernel_multi<P, T>), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &smooth_first_kernel<P, T>, grid_, block_, smem_, s_, NF, Dinv, b, xout, bh, omega, w, hnext, bout);
}


// Repack the FP64 operator (groups of 2) into another storage precision
// (groups of 16 / sizeof(TO)); padding lanes are zero.
template <typename TO>
__global__ void repack_kernel(const double *__restrict__ src, int ns, size_t NF, TO *__restrict__ dst) {
    constexpr int G = 16 / int(sizeof(TO));
    const size_t tid = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const size_t nq = (size_t(ns) + G - 1) / G;
    if (tid >= nq * NF) return;
    const size_t q = tid / NF, e = tid % NF;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const size_t j = q * G + g;
        double v = 0.0;
        if (j < size_t(ns)) v = src[((j / 2) * NF + e) * 2 + (j % 2)];
        dst[(q * NF + e) * G + g] = convert_to<TO>(v);
    }
}

// lambda layout [NF][PP] <-> internal [PP][NF]
__global__ void to_internal_kernel(int NF, int PP, const double *ext, double *in) {
    const size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= size_t(NF) * PP) return;
    const size_t e = i / PP, r = i % PP;
    in[r * NF + e] = ext[i];
}
__device__ __forceinline__ void to_external_kernel_impl(int bid_, int nb_, int NF, int PP, const double *in,
                                                        double *ext) {
    const size_t i = size_t(bid_) * blockDim.x + threadIdx.x;
    if (i >= size_t(NF) * PP) return;
    const size_t e = i / PP, r = i % PP;
    ext[i] = in[r * NF + e];
}
__global__ void to_external_kernel(int NF, int PP, const double *in, double *ext) {
    pdl_wait();
    to_external_kernel_impl(blockIdx.x, gridDim.x, NF, PP, in, ext);
}
struct to_external_kernel_args {
    int nb_;
    int NF;
    int PP;
    const double *in;
    double *ext;
};
__global__ void to_external_kernel_multi(const __grid_constant__ MultiP<to_external_kernel_args> M) {
    pdl_wait();
    int b_;
    const to_external_kernel_args &q_ = M.a[merge_find(M.start, M.n, b_)];
    to_external_kernel_impl(b_, q_.nb_, q_.NF, q_.PP, q_.in, q_.ext);
}
void to_external_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int NF, int PP,
                           const double *in, double *ext) {
    if (Recorder *r_ = batch_recorder()) {
        to_external_kernel_args q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.NF = NF;
        q_.PP = PP;
        q_.in = in;
        q_.ext = ext;
        batch_record(r_, reinterpret_cast<const void *>(&to_external_kernel_multi), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &to_external_kernel, grid_, block_, smem_, s_, NF, PP, in, ext);
}


// cell unknown kappa of cell K from the caller's r_u [N][2][NP], r_h [N][NP]
template <int NP>
__device__ __forceinline__ double cell_rhs(const double *r_u, const double *r_h, int K, int kap) {
    return kap < 2 * NP ? r_u[size_t(K) * 2 * NP + kap] : r_h[size_t(K) * NP + kap - 2 * NP];
}

// step 1, cell part: ycell[t][K] = sum_kappa W[t*NK + kappa][K] r_K[kappa]
template <int P>
__global__ void rhs_cell_kernel(int N, const double *__restrict__ W, const double *__restrict__ r_u,
                                const double *__restrict__ r_h, double *__restrict__ ycell) {
    constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2, NK = 3 * NP, M = 3 * PP;
    const size_t idx = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= size_t(N) * M) return;
    const int t = int(idx / N), K = int(idx % N);
    double acc = 0.0;
#pragma unroll 5
    for (int kap = 0; kap < NK; ++kap)
        acc = fma(__ldg(W + size_t(t * NK + kap) * N + K), cell_rhs<NP>(r_u, r_h, K, kap), acc);
    ycell[idx] = acc;
}

// g on facet e = the two cells' contributions (step 1 of Sec. 4.2); with
// partial non-null also ||g||^2 (block sums, the last block adding them in
// block order into out[0] and handing the value to the host through pub)
template <int P>
__device__ __forceinline__ void rhs_gather_kernel_impl(int bid_, int nb_, int N, int NF,
                                                       const double *__restrict__ ycell,
                                                       const int32_t *__restrict__ fcell,
                                                       const int32_t *__restrict__ fedge,
                                                       const int32_t *__restrict__ flip, double *__restrict__ g,
                                                       double *partial, unsigned int *counter, double *out,
                                                       HostValue *pub, int32_t seq, const F32Copy c32) {
    constexpr int PP = P + 1;
    const int e = bid_ * blockDim.x + threadIdx.x;
    double sq = 0.0;
    if (e < NF) {
        double v[PP];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int K = fcell[2 * e + s], i = fedge[2 * e + s], f = flip[3 * K + i];
#pragma unroll
            for (int r = 0; r < PP; ++r) {
                const double y = ycell[size_t(i * PP + (f ? P - r : r)) * N + K];
                v[r] = s == 0 ? y : v[r] + y;
            }
        }
#pragma unroll
        for (int r = 0; r < PP; ++r) {
            g[size_t(r) * NF + e] = v[r];
            sq = fma(v[r], v[r], sq);
        }
        if (c32.b32) {
#pragma unroll
            for (int r = 0; r < PP; ++r) {
                c32.b32[size_t(r) * NF + e] = to_float(mul_pow2(v[r], c32.scale));
                c32.z32[size_t(r) * NF + e] = 0.0f;
            }
        }
    }
    if (!partial) return;
    __shared__ bool last;
    const double tot = block_sum_warp0(sq);
    if (threadIdx.x == 0) {
        partial[bid_] = tot;
        __threadfence();                       // the partial is visible before the count
        last = atomicAdd(counter, 1u) == unsigned(nb_) - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double a = 0.0;
    for (int i = threadIdx.x; i < nb_; i += blockDim.x) a += partial[i];
    a = block_sum_warp0(a);
    if (threadIdx.x == 0) {
        *counter = 0u;
        out[0] = a;
        if (c32.root_a) *c32.root_a = sqrt(a) * c32.scale;
        if (c32.root_b) *c32.root_b = sqrt(a) * c32.scale;
        if (pub) {
            pub->v = a;
            __threadfence_system();
            *reinterpret_cast<volatile int32_t *>(&pub->seq) = seq;
        }
    }
}
template <int P>
__global__ void rhs_gather_kernel(int N, int NF, const double *__restrict__ ycell, const int32_t *__restrict__ fcell,
                                  const int32_t *__restrict__ fedge, const int32_t *__restrict__ flip,
                                  double *__restrict__ g, double *partial, unsigned int *counter, double *out,
                                  HostValue *pub, int32_t seq, const F32Copy c32) {
    pdl_wait();
    rhs_gather_kernel_impl<P>(blockIdx.x, gridDim.x, N, NF, ycell, fcell, fedge, flip, g, partial, counter, out, pub,
                              seq, c32);
}
template <int P>
struct rhs_gather_kernel_args {
    int nb_;
    int N;
    int NF;
    const double *ycell;
    const int32_t *fcell;
    const int32_t *fedge;
    const int32_t *flip;
    double *g;
    double *partial;
    unsigned int *counter;
    double *out;
    HostValue *pub;
    int32_t seq;
    F32Copy c32;
};
template <int P>
__global__ void rhs_gather_kernel_multi(const __grid_constant__ MultiP<rhs_gather_kernel_args<P>> M) {
    pdl_wait();
    int b_;
    const rhs_gather_kernel_args<P> &q_ = M.a[merge_find(M.start, M.n, b_)];
    rhs_gather_kernel_impl<P>(b_, q_.nb_, q_.N, q_.NF, q_.ycell, q_.fcell, q_.fedge, q_.flip, q_.g, q_.partial,
                              q_.counter, q_.out, q_.pub, q_.seq, q_.c32);
}
template <int P>
void rhs_gather_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int N, int NF,
                          const double *ycell, const int32_t *fcell, const int32_t *fedge, const int32_t *flip,
                          double *g, double *partial, unsigned int *counter, double *out, HostValue *pub,
                          int32_t seq, const F32Copy &c32) {
    if (Recorder *r_ = batch_recorder()) {
        rhs_gather_kernel_args<P> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.N = N;
        q_.NF = NF;
        q_.ycell = ycell;
        q_.fcell = fcell;
        q_.fedge = fedge;
        q_.flip = flip;
        q_.g = g;
        q_.partial = partial;
        q_.counter = counter;
        q_.out = out;
        q_.pub = pub;
        q_.seq = seq;
        q_.c32 = c32;
        batch_record(r_, reinterpret_cast<const void *>(&rhs_gather_kernel_multi<P>), q_, grid_, block_, smem_,
                     kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &rhs_gather_kernel<P>, grid_, block_, smem_, s_, N, NF, ycell, fcell, fedge, flip, g,
               partial, counter, out, pub, seq, c32);
}


// Step 3, q_K = R_M r_K - X_B lambda_K, by the rows of both (recover_by_rows in api.cu), one
// thread per row and cell.  A block takes whole cells and stages their r and lambda before it writes,
// so that u and h_out may be r_u and r_h, as in the kernels below.  Latency bounds it on small
// meshes: a thread issues the loads of its row of R_M first (512 cells with a cold cache, p = 1 .. 4:
// 5.6, 6.8, 8.2 and 11.4 us, instead of 6.8, 9.0, 13.8 and 18.2 with r and lambda read by every
// thread).  At p = 1, which takes it at every size, the FP64 pipe does, and seven blocks per SM
// instead of early loads: 34.6 us on 131,072 cells, 43.0 with them.
template <int P> constexpr int kRowCells = P == 1 ? 32 : P == 2 ? 16 : 8;
template <int P>
__global__ void __launch_bounds__(kRowCells<P> * 3 * (P + 1) * (P + 2) / 2, P == 1 ? 7 : 1)
    recover_rows_kernel(int N, int NF, const double *__restrict__ Rm, const double *__restrict__ Xb, const double *r_u,
                        const double *r_h, const double *__restrict__ lam, const int32_t *__restrict__ facet_of,
                        const int32_t *__restrict__ flip, double *u, double *hout) {
    constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2, NK = 3 * NP, M = 3 * PP, CC = kRowCells<P>, NT = CC * NK;
    __shared__ double sR[NK][CC + 1], sL[M][CC + 1];
    const int t = threadIdx.x, c = t % CC, rho = t / CC, K0 = blockIdx.x * CC, K = K0 + c, nc = min(CC, N - K0);
    const double *rm = Rm + size_t(rho) * NK * N + K, *xb = Xb + size_t(rho) * M * N + K;
    double a[NK];
    if (P > 1 && K < N) {
#pragma unroll
        for (int kap = 0; kap < NK; ++kap) a[kap] = __ldg(rm + size_t(kap) * N);
    }
    for (int j = t; j < nc * 2 * NP; j += NT) sR[j % (2 * NP)][j / (2 * NP)] = r_u[size_t(K0) * 2 * NP + j];
    for (int j = t; j < nc * NP; j += NT) sR[2 * NP + j % NP][j / NP] = r_h[size_t(K0) * NP + j];
    for (int j = t; j < nc * M; j += NT) {
        const int cell = j / M, q = j % M, i = q / PP, jj = q % PP;
        const int f = facet_of[3 * (K0 + cell) + i], fl = flip[3 * (K0 + cell) + i];
        sL[q][cell] = lam[size_t(fl ? P - jj : jj) * NF + f];
    }
    __syncthreads();
    if (K >= N) return;
    double acc = 0.0;
#pragma unroll
    for (int kap = 0; kap < NK; ++kap) acc = fma(P > 1 ? a[kap] : __ldg(rm + size_t(kap) * N), sR[kap][c], acc);
#pragma unroll
    for (int q = 0; q < M; ++q) acc = fma(-__ldg(xb + size_t(q) * N), sL[q][c], acc);
    if (rho < 2 * NP) u[size_t(K) * 2 * NP + rho] = acc;
    else hout[size_t(K) * NP + rho - 2 * NP] = acc;
}

// The same on larger meshes: h by the rows of R_M and X_B, the velocity from the
// momentum equations,
//   u = R w,   w = r_u - tau g (grad h + sum_e n_e lift_e (lambda - h)),   R = [P Q; -Q P],
// the weak gradient with the trace terms taken as the nodal one (whose vanishing entries are
// left out) plus the lifted jumps.  P and Q are numbers where f is constant on every cell
// (FC); else n_p x n_p matrices, kept as Q, P - Q and P + Q, so that R w takes three products,
//   k = Q (w_x + w_y),   u_x = (P - Q) w_x + k,   u_y = (P + Q) w_y - k.
// The FP64 pipe is the bound: at p = 3 about 860 (FC) and 1,120 FMAs per cell instead of
// the 1,260 of all rows of R_M and X_B: 192 instead of 314 us on 131,072 cells, 18.0 instead
// of 21.0 on 18,432 at p = 2; f varying 169 instead of 185 on 81,920.
// 32 cells per block (lane = cell), the warps take the nodes in turn.
template <int P> constexpr int kRecWarps = P == 2 ? 6 : 5;
template <int P, bool FC>
__global__ void __launch_bounds__(32 * kRecWarps<P>) recover_kernel(int N, int NF, const double *__restrict__ Rm,
                                                                            const double *__restrict__ Xb,
                                                                            const double *__restrict__ nref,
                                                                            const double *__restrict__ X,
                                                                            const double *__restrict__ fcell, double tau,
                                                                            double tg, const double *__restrict__ r_u,
                                                                            const double *__restrict__ r_h,
                                                                            const double *__restrict__ lam,
                                                                            const int32_t *__restrict__ facet_of,
                                                                            const int32_t *__restrict__ flip,
                                                                            double *__restrict__ u,
                                                                            double *__restrict__ hout) {
    constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2, NK = 3 * NP, M = 3 * PP, NW = kRecWarps<P>;
    constexpr NodalOffsets O = nodal_offsets(P);
    static_assert(NP % NW == 0, "every warp takes NP / NW nodes");
    __shared__ double sV[NK][33], sL[M][33], geo[12][32];      // r, then q; lambda, then the jumps; weights
    const int K0 = blockIdx.x * 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5, K = K0 + lane;
    const int nc = min(32, N - K0);
    for (int j = threadIdx.x; j < nc * 2 * NP; j += 32 * NW) sV[j % (2 * NP)][j / (2 * NP)] = r_u[size_t(K0) * 2 * NP + j];
    for (int j = threadIdx.x; j < nc * NP; j += 32 * NW) sV[2 * NP + j % NP][j / NP] = r_h[size_t(K0) * NP + j];
    for (int j = threadIdx.x; j < nc * M; j += 32 * NW) {
        const int cell = j / M, q = j % M, i = q / PP, jj = q % PP;
        const int f = facet_of[3 * (K0 + cell) + i], fl = flip[3 * (K0 + cell) + i];
        sL[q][cell] = lam[size_t(fl ? P - jj : jj) * NF + f];
    }
    const bool on = K < N;
    if (w == NW - 1 && on) {
        // tau g times J^-T (0..3) and n_e / det (4..9), then R (10, 11)
        const double *x = X + size_t(K) * 6;
        const double J00 = x[2] - x[0], J01 = x[4] - x[0], J10 = x[3] - x[1], J11 = x[5] - x[1];
        const double s = tg / (J00 * J11 - J01 * J10);
        geo[0][lane] = J11 * s;
        geo[1][lane] = -J10 * s;
        geo[2][lane] = -J01 * s;
        geo[3][lane] = J00 * s;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int v1 = (i + 1) % 3, v2 = (i + 2) % 3;
            geo[4 + 2 * i][lane] = s * (x[2 * v2 + 1] - x[2 * v1 + 1]);
            geo[5 + 2 * i][lane] = -s * (x[2 * v2] - x[2 * v1]);
        }
        const double f = tau * fcell[size_t(K) * 3], kap = 1.0 / fma(f, f, 1.0);
        geo[10][lane] = kap;
        geo[11][lane] = f * kap;
    }
    __syncthreads();
    double hv[NP / NW];
    if (on) {
#pragma unroll
        for (int t = 0; t < NP / NW; ++t) {
            const size_t i = size_t(w + t * NW);
            double acc = 0.0;
#pragma unroll 10
            for (int kap = 0; kap < NK; ++kap)
                acc = fma(__ldg(Rm + (rm_offsets(P, FC, false).h + i * NK + kap) * N + K), sV[kap][lane], acc);
#pragma unroll
            for (int q = 0; q < M; ++q) acc = fma(-__ldg(Xb + ((2 * NP + i) * M + q) * N + K), sL[q][lane], acc);
            hv[t] = acc;
        }
    }
    __syncthreads();                            // every warp has read r and lambda
    if (on) {
#pragma unroll
        for (int t = 0; t < NP / NW; ++t) sV[2 * NP + w + t * NW][lane] = hv[t];
    }
    __syncthreads();
    if (on)
        for (int q = w; q < M; q += NW) sL[q][lane] -= sV[2 * NP + edge_cell_node(P, q / PP, q % PP)][lane];
    __syncthreads();
    if (on) {
        static_for<NP>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if (i % NW != w) return;
            double dx = 0.0, dy = 0.0;
            static_for<NP>([&](auto kk) {
                constexpr int k = decltype(kk)::value;
                const double h = sV[2 * NP + k][lane];
                if constexpr (nodal_dx_nonzero(P, i, k)) dx = fma(__ldg(nref + O.Dx + i * NP + k), h, dx);
                if constexpr (nodal_dy_nonzero(P, i, k)) dy = fma(__ldg(nref + O.Dy + i * NP + k), h, dy);
            });
            double wx = sV[i][lane], wy = sV[NP + i][lane];
            wx = fma(-geo[0][lane], dx, fma(-geo[1][lane], dy, wx));
            wy = fma(-geo[2][lane], dx, fma(-geo[3][lane], dy, wy));
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                double l = 0.0;
#pragma unroll
                for (int jj = 0; jj < PP; ++jj) l = fma(__ldg(nref + O.lift + (e * NP + i) * PP + jj), sL[e * PP + jj][lane], l);
                wx = fma(-geo[4 + 2 * e][lane], l, wx);
                wy = fma(-geo[5 + 2 * e][lane], l, wy);
            }
            if constexpr (FC) {
                const double kap = geo[10][lane], fk = geo[11][lane];
                sV[i][lane] = fma(kap, wx, fk * wy);
                sV[NP + i][lane] = fma(kap, wy, -fk * wx);
            } else {
                sV[i][lane] = wx;
                sV[NP + i][lane] = wy;
            }
        });
    }
    __syncthreads();
    if constexpr (!FC) {
        if (on)
            for (int i = w; i < NP; i += NW) sL[i][lane] = sV[i][lane] + sV[NP + i][lane];   // (the jumps have been read)
        __syncthreads();
        double ux[NP / NW], uy[NP / NW];
        if (on) {
#pragma unroll
            for (int t = 0; t < NP / NW; ++t) {
                const size_t i = size_t(w + t * NW), NN = NP * NP;
                double a = 0.0, b = 0.0, c = 0.0;
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    c = fma(__ldg(Rm + (i * NP + k) * N + K), sL[k][lane], c);
                    a = fma(__ldg(Rm + (NN + i * NP + k) * N + K), sV[k][lane], a);
                    b = fma(__ldg(Rm + (2 * NN + i * NP + k) * N + K), sV[NP + k][lane], b);
                }
                ux[t] = a + c;
                uy[t] = b - c;
            }
        }
        __syncthreads();                        // every warp has read w
        if (on) {
#pragma unroll
            for (int t = 0; t < NP / NW; ++t) {
                sV[w + t * NW][lane] = ux[t];
                sV[NP + w + t * NW][lane] = uy[t];
            }
        }
        __syncthreads();
    }
    for (int j = threadIdx.x; j < nc * 2 * NP; j += 32 * NW) u[size_t(K0) * 2 * NP + j] = sV[j % (2 * NP)][j / (2 * NP)];
    for (int j = threadIdx.x; j < nc * NP; j += 32 * NW) hout[size_t(K0) * NP + j] = sV[2 * NP + j % NP][j / NP];
}

// P1 restriction rho = pi^T: r_c[v] = sum over facet ends at v of the nodal
// weights of the linear interpolant (1 - t_r at the lower vertex, t_r at the higher).
// Latency bounds it (list, facet id, p + 1 values, one after the other), so in FP32 eight
// lanes (L) share a vertex's facet ends up to kRestrictShared vertices (1.3 times the threads
// that 152 SMs hold; a line between the measured 40,962 and 65,536): 5.4 instead of 6.5 us for
// 40,962 vertices at p = 3, 3.4 instead of 3.7 for 20,736 at p = 2, but 6.5 instead of 5.3 for
// 65,536 and 12.0 instead of 7.8 for 163,842.  In FP64, where the lanes' additions would take
// the pipe longer than the loads, and on the larger meshes one thread takes them all.
constexpr int kRestrictShared = 49152;
template <int P, typename T, int L>
__device__ __forceinline__ void restrict_kernel_impl(int bid_, int nb_, int nv, int NF,
                                                     const int32_t *__restrict__ v2f_ptr,
                                                     const int32_t *__restrict__ v2f, const T *__restrict__ r,
                                                     T *__restrict__ rc, const T *__restrict__ dinv0, T omega,
                                                     T *__restrict__ x0) {
    const int t = bid_ * blockDim.x + threadIdx.x, v = t / L, q = t % L;
    T acc = T(0);
    if (v < nv) {
        const int k1 = v2f_ptr[v + 1];
        for (int k = v2f_ptr[v] + q; k < k1; k += L) {
            const int code = v2f[k], e = code >> 1, hi = code & 1;
#pragma unroll
            for (int j = 0; j <= P; ++j) {
                const T w = T(j) / T(P);
                acc = fma(hi ? w : T(1) - w, r[size_t(j) * NF + e], acc);
            }
        }
    }
#pragma unroll
    for (int off = L / 2; off > 0; off /= 2) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (v >= nv || q != 0) return;
    rc[v] = acc;
    // first damped Jacobi sweep of the P1 level from zero, fused (x0 may be null)
    if (x0) x0[v] = omega * dinv0[v] * acc;
}
template <int P, typename T, int L>
__global__ void restrict_kernel(int nv, int NF, const int32_t *__restrict__ v2f_ptr, const int32_t *__restrict__ v2f,
                                const T *__restrict__ r, T *__restrict__ rc, const T *__restrict__ dinv0, T omega,
                                T *__restrict__ x0) {
    pdl_wait();
    restrict_kernel_impl<P, T, L>(blockIdx.x, gridDim.x, nv, NF, v2f_ptr, v2f, r, rc, dinv0, omega, x0);
}
template <int P, typename T, int L>
struct restrict_kernel_args {
    int nb_;
    int nv;
    int NF;
    const int32_t *v2f_ptr;
    const int32_t *v2f;
    const T *r;
    T *rc;
    const T *dinv0;
    T omega;
    T *x0;
};
template <int P, typename T, int L>
__global__ void restrict_kernel_multi(const __grid_constant__ MultiP<restrict_kernel_args<P, T, L>> M) {
    pdl_wait();
    int b_;
    const restrict_kernel_args<P, T, L> &q_ = M.a[merge_find(M.start, M.n, b_)];
    restrict_kernel_impl<P, T, L>(b_, q_.nb_, q_.nv, q_.NF, q_.v2f_ptr, q_.v2f, q_.r, q_.rc, q_.dinv0, q_.omega, q_.x0);
}
template <int P, typename T, int L>
void restrict_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int nv, int NF,
                        const int32_t *v2f_ptr, const int32_t *v2f, const T *r, T *rc, const T *dinv0, T omega,
                        T *x0) {
    if (Recorder *r_ = batch_recorder()) {
        restrict_kernel_args<P, T, L> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.nv = nv;
        q_.NF = NF;
        q_.v2f_ptr = v2f_ptr;
        q_.v2f = v2f;
        q_.r = r;
        q_.rc = rc;
        q_.dinv0 = dinv0;
        q_.omega = omega;
        q_.x0 = x0;
        batch_record(r_, reinterpret_cast<const void *>(&restrict_kernel_multi<P, T, L>), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &restrict_kernel<P, T, L>, grid_, block_, smem_, s_, nv, NF, v2f_ptr, v2f, r, rc, dinv0, omega, x0);
}


// x += pi e_c (linear interpolation along each facet)
template <int P, typename T>
__global__ void prolong_add_kernel(int NF, const int32_t *__restrict__ fverts, const T *__restrict__ ec,
                                   T *__restrict__ x) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NF) return;
    const T a = ec[fverts[2 * e]], b = ec[fverts[2 * e + 1]];
#pragma unroll
    for (int j = 0; j <= P; ++j) {
        const T t = T(j) / T(P);
        x[size_t(j) * NF + e] += (T(1) - t) * a + t * b;
    }
}

inline unsigned blocks(size_t n, int bs) { return unsigned((n + bs - 1) / bs); }


}  // namespace

// operators by type: S, the inverse diagonal blocks, and the sweeps' H and D (null where the
// sweeps of that type take S; HDG_MIXED_BF16 keeps H in BF16)
template <typename T> struct Ops;
template <> struct Ops<double> {
    static const double *S(hdg_handle *h) { return h->d_Sval; }
    static const double *D(hdg_handle *h) { return h->d_Dinv; }
    static const double *H(hdg_handle *h) { return h->d_H; }
    static const double *Dg(hdg_handle *h) { return h->d_D; }
};
template <> struct Ops<float> {
    static const float *S(hdg_handle *h) { return h->d_Sval32; }
    static const float *D(hdg_handle *h) { return h->d_Dinv32; }
    static const float *H(hdg_handle *h) { return h->d_H32; }
    static const float *Dg(hdg_handle *h) { return h->d_D32; }
};
inline bool bf16_pre(hdg_handle *h) { return h->prm.precision == HDG_MIXED_BF16 && h->d_H16; }

template <typename T, int B>
cudaError_t apply_dots_b(hdg_handle *h, unsigned nb, const T *x, T *y, const T *V, size_t ld, int k, double *partial,
                         unsigned int *counter, double *hdots, T *hneg) {
    constexpr int BB = sizeof(T) == 8 ? 4 : B;
    HDG_DISPATCH_PF(h->pf, T, (apply_dots_kernel_go<P, T, T, BB>(nb, 256, 0, h->stream, 
                             h->NF, Ops<T>::S(h), h->d_nbr, x, y, V, ld, k, partial, counter, hdots, hneg)));
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_apply_dots_t(hdg_handle *h, const T *x, T *y, const T *V, size_t ld, int k, double *partial,
                                unsigned int *counter, double *hdots, T *hneg) {
    // Blocks per SM that the kernel is compiled for: fewer leave a thread the registers for
    // more loads in flight (FP32, 4: eight vectors at a time instead of four), more finish
    // the grid in fewer rounds.  A round of 4, 5 and 6 blocks per SM takes about 8, 9.5 and
    // 10.5 us (p = 2, 491,520 facets: 4, 3 and 3 rounds, 31.3, 28.9 and 31.5 us; p = 3,
    // 196,608: 2, 2 and 1 round, 16.5, 18.3 and 14.9; p = 4, 30,000: one, 8.7, 10.9 and
    // 11.7).  FP64: bound by its pipe, four.
    const unsigned nb = blocks(h->NF, 256);
    auto rounds = [&](unsigned b) { return (nb + 152 * b - 1) / (152 * b); };
    int B = 4;
    if (sizeof(T) == 4) {
        const unsigned c4 = 16 * rounds(4), c5 = 19 * rounds(5), c6 = 21 * rounds(6);
        B = c4 <= c5 && c4 <= c6 ? 4 : c5 <= c6 ? 5 : 6;
    }
    switch (B) {
        case 4: return apply_dots_b<T, 4>(h, nb, x, y, V, ld, k, partial, counter, hdots, hneg);
        case 5: return apply_dots_b<T, 5>(h, nb, x, y, V, ld, k, partial, counter, hdots, hneg);
        default: return apply_dots_b<T, 6>(h, nb, x, y, V, ld, k, partial, counter, hdots, hneg);
    }
}
template <typename T>
cudaError_t launch_apply_t(hdg_handle *h, const T *x, T *y) {
    HDG_DISPATCH_PF(h->pf, T, (apply_kernel<P, T, T><<<blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream>>>(h->NF, Ops<T>::S(h), h->d_nbr, x, y)));
    return cudaGetLastError();
}
// res = b - S x, for the preconditioner and the Krylov residual
template <typename T>
cudaError_t launch_residual_t(hdg_handle *h, const T *b, const T *x, T *r) {
    HDG_DISPATCH_PF(h->pf, T, (residual_kernel_go<P, T, T>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, Ops<T>::S(h), h->d_nbr, b, x, r)));
    return cudaGetLastError();
}
// A sweep with b = D^-1 times the right-hand side where the handle's sweeps of this type
// work on D^-1 S (hat_form), else the right-hand side itself; with cheb, a step of the
// Chebyshev iteration xout = x + omega D^-1 (b - S x) + beta (x - xprev)
template <typename T, bool CHEB>
cudaError_t smooth_any(hdg_handle *h, const T *b, const T *x, T *xout, T om, T beta, const T *xprev) {
    if constexpr (std::is_same<T, float>::value) if (bf16_pre(h)) {
        HDG_DISPATCH_PF(h->pf, T, (smooth_kernel_go<P, T, __nv_bfloat16, true, CHEB>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, h->d_H16, nullptr, h->d_nbr, b, x, xout, om, beta, xprev)));
        return cudaGetLastError();
    }
    if (Ops<T>::H(h)) {
        HDG_DISPATCH_PF(h->pf, T, (smooth_kernel_go<P, T, T, true, CHEB>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, Ops<T>::H(h), nullptr, h->d_nbr, b, x, xout, om, beta, xprev)));
    } else {
        HDG_DISPATCH_PF(h->pf, T, (smooth_kernel_go<P, T, T, false, CHEB>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, Ops<T>::S(h), Ops<T>::D(h), h->d_nbr, b, x, xout, om, beta, xprev)));
    }
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_smooth_t(hdg_handle *h, const T *b, const T *x, T *xout) {
    return smooth_any<T, false>(h, b, x, xout, T(h->prm.omega), T(0), nullptr);
}
template <typename T>
cudaError_t launch_smooth_cheb_t(hdg_handle *h, const T *b, const T *x, T *xout, double omega, double beta,
                                 const T *xprev) {
    return smooth_any<T, true>(h, b, x, xout, T(omega), T(beta), xprev);
}
template <typename T>
cudaError_t launch_smooth_first_t(hdg_handle *h, const T *b, T *x, T *bh, const T *w, const double *hnext, T *bout,
                                  double omega) {
    const T om = T(omega > 0 ? omega : h->prm.omega);
    HDG_DISPATCH_PF(h->pf, T, (smooth_first_kernel_go<P, T>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, Ops<T>::D(h), b, x, bh, om, w, hnext, bout)));
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_restrict_t(hdg_handle *h, const T *r, T *rc, const T *dinv0, T omega, T *x0) {
    if (sizeof(T) == 4 && h->nv <= kRestrictShared) {
        HDG_DISPATCH_P(h->p, (restrict_kernel_go<P, T, sizeof(T) == 4 ? 8 : 1>(blocks(size_t(h->nv) * 8, 256), 256, 0, h->stream, h->nv, h->NF, h->d_v2f_ptr, h->d_v2f, r, rc, dinv0, omega, x0)));
        return cudaGetLastError();
    }
    HDG_DISPATCH_P(h->p, (restrict_kernel_go<P, T, 1>(blocks(h->nv, 256), 256, 0, h->stream, h->nv, h->NF, h->d_v2f_ptr, h->d_v2f, r, rc, dinv0, omega, x0)));
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_smooth_prolong_t(hdg_handle *h, const T *ec, const T *y, const T *x, T *xout, double omega,
                                    T *x0out) {
    const T om = T(omega > 0 ? omega : h->prm.omega);
    const T *q;
    if constexpr (std::is_same<T, float>::value) q = h->d_Q32;
    else q = h->d_Q;
    if (x0out) {
        HDG_DISPATCH_P(h->p, (smooth_prolong_kernel_go<P, T, true>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, q, h->d_facet_verts, h->d_facet_opp, ec, y, x, xout, om, x0out)));
    } else {
        HDG_DISPATCH_P(h->p, (smooth_prolong_kernel_go<P, T>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, q, h->d_facet_verts, h->d_facet_opp, ec, y, x, xout, om, nullptr)));
    }
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_residual_smooth_t(hdg_handle *h, const T *b, const T *x, T *res, T *y, double omega) {
    const T om = T(omega > 0 ? omega : h->prm.omega);
    if constexpr (std::is_same<T, float>::value) if (bf16_pre(h)) {
        HDG_DISPATCH_P(h->p, (residual_smooth_kernel_go<P, T, __nv_bfloat16, true>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, h->d_H16, Ops<T>::Dg(h), h->d_nbr, b, x, res, y, om)));
        return cudaGetLastError();
    }
    if (Ops<T>::H(h)) {
        HDG_DISPATCH_P(h->p, (residual_smooth_kernel_go<P, T, T, true>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, Ops<T>::H(h), Ops<T>::Dg(h), h->d_nbr, b, x, res, y, om)));
    } else {
        HDG_DISPATCH_P(h->p, (residual_smooth_kernel_go<P, T, T, false>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->NF, Ops<T>::S(h), Ops<T>::D(h), h->d_nbr, b, x, res, y, om)));
    }
    return cudaGetLastError();
}
template cudaError_t launch_residual_smooth_t<double>(hdg_handle *, const double *, const double *, double *, double *, double);
template cudaError_t launch_residual_smooth_t<float>(hdg_handle *, const float *, const float *, float *, float *, double);
template <typename T>
cudaError_t launch_prolong_add_t(hdg_handle *h, const T *ec, T *x) {
    HDG_DISPATCH_P(h->p, (prolong_add_kernel<P, T><<<blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream>>>(h->NF, h->d_facet_verts, ec, x)));
    return cudaGetLastError();
}
// FP32 copies of the packed FP64 operator and the inverse blocks
cudaError_t launch_repack(hdg_handle *h) {
    const int pp = h->pp, ns = 5 * pp * pp, nd = pp * pp;
    const size_t NF = h->NF;
    auto nq = [&](int n, int G) { return (size_t(n) + G - 1) / G * NF; };
    if (h->d_Sval32) {
        repack_kernel<float><<<blocks(nq(ns, 4), 256), 256, 0, h->stream>>>(h->d_Sval, ns, NF, h->d_Sval32);
        repack_kernel<float><<<blocks(nq(nd, 4), 256), 256, 0, h->stream>>>(h->d_Dinv, nd, NF, h->d_Dinv32);
    }
    return cudaGetLastError();
}

template cudaError_t launch_apply_t<double>(hdg_handle *, const double *, double *);
template cudaError_t launch_apply_dots_t<double>(hdg_handle *, const double *, double *, const double *, size_t, int,
                                                 double *, unsigned int *, double *, double *);
template cudaError_t launch_apply_dots_t<float>(hdg_handle *, const float *, float *, const float *, size_t, int,
                                                double *, unsigned int *, double *, float *);
template cudaError_t launch_apply_t<float>(hdg_handle *, const float *, float *);
template cudaError_t launch_residual_t<double>(hdg_handle *, const double *, const double *, double *);
template cudaError_t launch_residual_t<float>(hdg_handle *, const float *, const float *, float *);
template cudaError_t launch_smooth_t<double>(hdg_handle *, const double *, const double *, double *);
template cudaError_t launch_smooth_t<float>(hdg_handle *, const float *, const float *, float *);
template cudaError_t launch_smooth_cheb_t<double>(hdg_handle *, const double *, const double *, double *, double,
                                                  double, const double *);
template cudaError_t launch_smooth_cheb_t<float>(hdg_handle *, const float *, const float *, float *, double, double,
                                                 const float *);
template cudaError_t launch_smooth_first_t<double>(hdg_handle *, const double *, double *, double *, const double *,
                                                   const double *, double *, double);
template cudaError_t launch_smooth_first_t<float>(hdg_handle *, const float *, float *, float *, const float *, const double *,
                                                  float *, double);
template cudaError_t launch_restrict_t<double>(hdg_handle *, const double *, double *, const double *, double, double *);
template cudaError_t launch_restrict_t<float>(hdg_handle *, const float *, float *, const float *, float, float *);
cudaError_t launch_hat_op(hdg_handle *h) {
    const HatOut o{h->d_H, h->d_D, h->d_Q, h->d_H32, h->d_D32, h->d_Q32, h->d_H16};
    const unsigned nb = blocks(h->NF, 128);
    if (h->d_Q) {
        HDG_DISPATCH_P(h->p, (hat_op_kernel<P, true><<<nb, 128, 0, h->stream>>>(h->NF, h->d_Sval, h->d_Dinv, h->d_nbr,
                                                                              h->d_facet_verts, o)));
    } else {
        HDG_DISPATCH_PF(h->pf, double, (hat_op_kernel<P, false><<<nb, 128, 0, h->stream>>>(h->NF, h->d_Sval, h->d_Dinv,
                                                                                         h->d_nbr, h->d_facet_verts, o)));
    }
    return cudaGetLastError();
}
template cudaError_t launch_smooth_prolong_t<double>(hdg_handle *, const double *, const double *, const double *, double *,
                                                     double, double *);
template cudaError_t launch_smooth_prolong_t<float>(hdg_handle *, const float *, const float *, const float *, float *,
                                                    double, float *);
template cudaError_t launch_prolong_add_t<double>(hdg_handle *, const double *, double *);
template cudaError_t launch_prolong_add_t<float>(hdg_handle *, const float *, float *);

cudaError_t launch_to_internal(hdg_handle *h, const double *ext, double *in) {
    size_t n = size_t(h->NF) * h->pp;
    to_internal_kernel<<<blocks(n, 256), 256, 0, h->stream>>>(h->NF, h->pp, ext, in);
    return cudaGetLastError();
}
cudaError_t launch_to_external(hdg_handle *h, const double *in, double *ext) {
    size_t n = size_t(h->NF) * h->pp;
    to_external_kernel_go(blocks(n, 256), 256, 0, h->stream, h->NF, h->pp, in, ext);
    return cudaGetLastError();
}

cudaError_t launch_rhs_gather(hdg_handle *h, const double *ycell, double *g, const NormOut &nrm) {
    HDG_DISPATCH_P(h->p, (rhs_gather_kernel_go<P>(blocks(h->NF, h->bs_facet), h->bs_facet, 0, h->stream, h->N, h->NF,
                                                  ycell, h->d_facet_cell, h->d_facet_edge, h->d_flip, g, nrm.partial,
                                                  nrm.counter, nrm.out, nrm.pub, nrm.seq, nrm.f32)));
    return cudaGetLastError();
}

cudaError_t launch_rhs(hdg_handle *h, const double *r_u, const double *r_h, double *g, double *ycell,
                       const NormOut &nrm) {
    if (h->prm.flux == 1) return nrm.partial ? cudaErrorInvalidValue : launch_rhs_lf(h, r_u, r_h, g, ycell);
    if (mode_ff(h->prm)) return launch_rhs_z(h, r_u, r_h, g, ycell, nullptr, nullptr, nullptr, nrm);
    size_t n = size_t(h->N) * h->m;
    HDG_DISPATCH_P(h->p, (rhs_cell_kernel<P><<<blocks(n, 256), 256, 0, h->stream>>>(h->N, h->d_W, r_u, r_h, ycell)));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_rhs_gather(h, ycell, g, nrm);
}

cudaError_t launch_recover(hdg_handle *h, const double *r_u, const double *r_h, const double *lam, double *u,
                           double *hout) {
    if (h->prm.flux == 1) return launch_recover_lf(h, r_u, r_h, lam, u, hout);
    if (h->rec_rows) {
        HDG_DISPATCH_P(h->p, (recover_rows_kernel<P><<<blocks(h->N, kRowCells<P>), kRowCells<P> * h->nK, 0, h->stream>>>(
                                 h->N, h->NF, h->d_Rm, h->d_Xb, r_u, r_h, lam, h->d_facet_of, h->d_flip, u, hout)));
        return cudaGetLastError();
    }
    const unsigned nb = blocks(h->N, 32);
    const double tau = h->prm.tau, tg = tau * h->prm.g;
    auto momentum = [&](auto kernel, int warps) {
        kernel<<<nb, 32 * warps, 0, h->stream>>>(h->N, h->NF, h->d_Rm, h->d_Xb, h->d_nref, h->d_X, h->d_fcell, tau, tg,
                                                 r_u, r_h, lam, h->d_facet_of, h->d_flip, u, hout);
    };
    switch (h->p) {
        case 2: h->f_const ? momentum(&recover_kernel<2, true>, kRecWarps<2>) : momentum(&recover_kernel<2, false>, kRecWarps<2>); break;
        case 3: h->f_const ? momentum(&recover_kernel<3, true>, kRecWarps<3>) : momentum(&recover_kernel<3, false>, kRecWarps<3>); break;
        case 4: h->f_const ? momentum(&recover_kernel<4, true>, kRecWarps<4>) : momentum(&recover_kernel<4, false>, kRecWarps<4>); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace hdg
