// Two-float arithmetic for the FP64 steps of the mixed-precision path: the
// condensed right-hand side (step 1 of the Schur-complement solve, Sec. 3.3),
// the refinement residual g - S lambda (Eq. schur_system) and the recovery of
// the cell unknowns (step 3).  GB300's FP64 pipe is far slower than its FP32
// one, and these steps are FP64-FMA bound there, not HBM bound.
//
// Every stored FP64 matrix entry a is kept as a pair (hi, lo) = (rn(a),
// rn(a - hi)) of floats (8 bytes, like the double), every FP64 input is split
// the same way once per use, and a sum of products is carried as
//   s + c:  s the running sum of the rounded leading products hi_a*hi_x, added
//           by error-free TwoSum steps; c the float sum of the exact product
//           errors (by FMA), the cross terms hi_a*lo_x + lo_a*hi_x and the
//           TwoSum errors.
// The dropped lo_a*lo_x and the rounding of c leave a relative error of about
// n * 2^-48 of sum |a_i x_i| (FP64: n * 2^-53), at a dozen FP32 operations per
// term.  Values must lie in the FP32 range (|v| < 3e38); an overflow shows up
// as Inf/NaN in the refinement residual, which the solver reports.
#include "common.h"

namespace hdg {

// launch family of this file for pdl_launch (facet-row kernels); the kernel
// that ends an inner solve goes with the Krylov kernels
constexpr unsigned kPdlFamily = 1;
constexpr unsigned kPdlKrylov = 4;

namespace {

inline unsigned blocks(size_t n, int bs) { return unsigned((n + bs - 1) / bs); }

// The cell kernels take 32 consecutive cells per block (lane = cell): the
// cells' right-hand sides r_K = (r_u, r_h) are read as contiguous chunks,
// split once into shared memory and shared by the warps, which take the output
// rows in turn; per-cell matrices are float pairs of two row entries in tiles of 32 cells
// ([tile][row][col pair][32], ff_pair_index, written by the condensation) and load
// coalesced, 16 bytes per lane.
constexpr int kCells = kFFCells;
constexpr int kCellsPad = kCells + 1;

// (n even: whole 16-byte groups of the packed operator; two groups per thread)
__global__ void split_kernel(const double2 *__restrict__ a, float4 *__restrict__ out, size_t n2) {
    const size_t i = size_t(blockIdx.x) * blockDim.x * 2 + threadIdx.x;
    double2 v[2];
#pragma unroll
    for (int u = 0; u < 2; ++u)
        if (i + u * blockDim.x < n2) v[u] = a[i + u * blockDim.x];
#pragma unroll
    for (int u = 0; u < 2; ++u)
        if (i + u * blockDim.x < n2) {
            const float2 x = split(v[u].x), y = split(v[u].y);
            out[i + u * blockDim.x] = make_float4(x.x, x.y, y.x, y.y);
        }
}

// acc += sum over the NCOL entries of one row (pairs p[cp * kCells], cp <
// (NCOL + 1) / 2, within the cell's tile) times x[col][lane], in column order
template <int NCOL>
__device__ __forceinline__ void row_pairs(FFAcc &acc, const float4 *__restrict__ p, const float2 (*x)[kCellsPad],
                                          int lane, bool negate = false) {
    constexpr int CP = (NCOL + 1) / 2;
#pragma unroll 3
    for (int cp = 0; cp < CP; ++cp) {
        const float4 v = __ldg(p + size_t(cp) * kCells);
        const float2 a0 = negate ? make_float2(-v.x, -v.y) : make_float2(v.x, v.y);
        acc.add(a0, x[2 * cp][lane]);
        if (2 * cp + 1 < NCOL) {
            const float2 a1 = negate ? make_float2(-v.z, -v.w) : make_float2(v.z, v.w);
            acc.add(a1, x[2 * cp + 1][lane]);
        }
    }
}

// The refinement iterate lambda is kept only as float pairs (hi, lo), the form
// the residual kernel reads; the correction x += scale * d then runs on the
// FP32 pipe, and the pairs are joined into FP64 once, when the solve ends.
// (hi, lo) += (sh + sl) * d, (sh, sl) = split(scale) formed once per block:
// the leading product by FMA with its exact error, the cross term sl * d, a
// TwoSum of the leading parts, the trailing parts added to its error and a
// renormalisation (about 2^-46 relative).  first: the iterate is zero and not
// read.
__device__ __forceinline__ float2 ff_add_scaled(float2 xv, float2 sc, float di, bool first) {
    const float ph = __fmul_rn(sc.x, di);
    const float pl = __fmaf_rn(sc.y, di, __fmaf_rn(sc.x, di, -ph));
    if (first) {
        const float t = __fadd_rn(ph, pl);
        return make_float2(t, __fsub_rn(pl, __fsub_rn(t, ph)));
    }
    const float t = __fadd_rn(xv.x, ph);
    const float bp = __fsub_rn(t, xv.x);
    float e = __fadd_rn(__fsub_rn(xv.x, __fsub_rn(t, bp)), __fsub_rn(ph, bp));
    e = __fadd_rn(e, __fadd_rn(xv.y, pl));
    const float hi = __fadd_rn(t, e);
    return make_float2(hi, __fsub_rn(e, __fsub_rn(hi, t)));
}
__device__ __forceinline__ void ff_axpy_kernel_impl(int bid_, int nb_, float2 *__restrict__ x2,
                                                    const float *__restrict__ d, const double *__restrict__ scale,
                                                    size_t n, int first) {
    // the entry's loads are issued before the block waits for the split scale
    const size_t i = size_t(bid_) * blockDim.x + threadIdx.x;
    const bool on = i < n;
    const float di = on ? d[i] : 0.0f;
    const float2 xv = on && !first ? x2[i] : make_float2(0.0f, 0.0f);
    __shared__ float2 sc;
    if (threadIdx.x == 0) sc = split(scale[0]);
    __syncthreads();
    if (!on) return;
    x2[i] = ff_add_scaled(xv, sc, di, first != 0);
}
__global__ void ff_axpy_kernel(float2 *__restrict__ x2, const float *__restrict__ d, const double *__restrict__ scale,
                               size_t n, int first) {
    pdl_wait();
    ff_axpy_kernel_impl(blockIdx.x, gridDim.x, x2, d, scale, n, first);
}
struct ff_axpy_kernel_args {
    int nb_;
    float2 *x2;
    const float *d;
    const double *scale;
    size_t n;
    int first;
};
__global__ void ff_axpy_kernel_multi(const __grid_constant__ MultiP<ff_axpy_kernel_args> M) {
    pdl_wait();
    int b_;
    const ff_axpy_kernel_args &q_ = M.a[merge_find(M.start, M.n, b_)];
    ff_axpy_kernel_impl(b_, q_.nb_, q_.x2, q_.d, q_.scale, q_.n, q_.first);
}
void ff_axpy_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, float2 *x2, const float *d,
                       const double *scale, size_t n, int first) {
    if (Recorder *r_ = batch_recorder()) {
        ff_axpy_kernel_args q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.x2 = x2;
        q_.d = d;
        q_.scale = scale;
        q_.n = n;
        q_.first = first;
        batch_record(r_, reinterpret_cast<const void *>(&ff_axpy_kernel_multi), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &ff_axpy_kernel, grid_, block_, smem_, s_, x2, d, scale, n, first);
}

// The end of the last cycle of an inner solve of the mixed refinement, in one
// pass: y = R^-1 s for the leading k x k triangle of the rotated Hessenberg
// matrix (column-major, leading dimension ldh), solved by one warp of every
// block with the substitution of the separate triangular-solve kernel; d = x +
// sum_c y_c Z_c with the FP32 sums of the separate basis update (x null: the
// inner iterate is still zero); then the refinement iterate's pairs +=
// scale[0] * d as ff_axpy forms it (first: pairs = scale[0] * d).  The same
// values as those three kernels, bit for bit.  Each thread takes kFinU entries
// a block width apart.
constexpr int kFinU = 8;
__device__ __forceinline__ void ff_finish_kernel_impl(int bid_, int nb_, const double *__restrict__ Hm, int ldh,
                                                      const double *__restrict__ sv, int k,
                                                      const float *__restrict__ Z, size_t ld,
                                                      const float *__restrict__ x, float2 *__restrict__ x2,
                                                      const double *__restrict__ scale, size_t n, int first) {
    extern __shared__ double R[];          // k x k, R[i * k + l] = row i, column l
    __shared__ double sS[64], yS[64];
    __shared__ float cf[64];
    __shared__ float2 sc;
    __shared__ double scl;
    if (threadIdx.x == 0) scl = scale[0];
    // the entries' x first (they do not wait for y)
    const size_t base = size_t(bid_) * blockDim.x * kFinU + threadIdx.x;
    float acc[kFinU];
#pragma unroll
    for (int u = 0; u < kFinU; ++u) {
        const size_t i = base + size_t(u) * blockDim.x;
        acc[u] = (x && i < n) ? x[i] : 0.0f;
    }
    for (int t = threadIdx.x; t < k * k; t += blockDim.x) {
        const int l = t / k, i = t % k;            // column l, row i
        if (i <= l) R[i * k + l] = Hm[size_t(l) * ldh + i];
    }
    for (int i = threadIdx.x; i < k; i += blockDim.x) sS[i] = sv[i];
    __syncthreads();
    if (threadIdx.x < 32) hess_back_substitute(R, sS, yS, k);
    else if (threadIdx.x == 32) sc = split(scl);
    __syncthreads();
    for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = float(1.0 * yS[i]);
    __syncthreads();
    // basis vector by basis vector, kFinU independent loads each and two
    // vectors' loads in flight (each entry still adds its terms in the order
    // c = 0, 1, ...)
#pragma unroll 2
    for (int c = 0; c < k; ++c) {
        const float cc = cf[c];
        const float *Zc = Z + size_t(c) * ld;
#pragma unroll
        for (int u = 0; u < kFinU; ++u) {
            const size_t i = base + size_t(u) * blockDim.x;
            if (i < n) acc[u] = fma(cc, Zc[i], acc[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < kFinU; ++u) {
        const size_t i = base + size_t(u) * blockDim.x;
        if (i < n) x2[i] = ff_add_scaled(first ? make_float2(0.0f, 0.0f) : x2[i], sc, acc[u], first != 0);
    }
}
__global__ void __launch_bounds__(256, 4) ff_finish_kernel(const double *__restrict__ Hm, int ldh,
                                                        const double *__restrict__ sv, int k,
                                                        const float *__restrict__ Z, size_t ld,
                                                        const float *__restrict__ x, float2 *__restrict__ x2,
                                                        const double *__restrict__ scale, size_t n, int first) {
    pdl_wait();
    ff_finish_kernel_impl(blockIdx.x, gridDim.x, Hm, ldh, sv, k, Z, ld, x, x2, scale, n, first);
}
struct ff_finish_kernel_args {
    int nb_;
    const double *Hm;
    int ldh;
    const double *sv;
    int k;
    const float *Z;
    size_t ld;
    const float *x;
    float2 *x2;
    const double *scale;
    size_t n;
    int first;
};
__global__ void __launch_bounds__(256, 4) ff_finish_kernel_multi(const __grid_constant__ MultiP<ff_finish_kernel_args> M) {
    pdl_wait();
    int b_;
    const ff_finish_kernel_args &q_ = M.a[merge_find(M.start, M.n, b_)];
    ff_finish_kernel_impl(b_, q_.nb_, q_.Hm, q_.ldh, q_.sv, q_.k, q_.Z, q_.ld, q_.x, q_.x2, q_.scale, q_.n, q_.first);
}
void ff_finish_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, const double *Hm, int ldh,
                         const double *sv, int k, const float *Z, size_t ld, const float *x, float2 *x2,
                         const double *scale, size_t n, int first) {
    if (Recorder *r_ = batch_recorder()) {
        ff_finish_kernel_args q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.Hm = Hm;
        q_.ldh = ldh;
        q_.sv = sv;
        q_.k = k;
        q_.Z = Z;
        q_.ld = ld;
        q_.x = x;
        q_.x2 = x2;
        q_.scale = scale;
        q_.n = n;
        q_.first = first;
        batch_record(r_, reinterpret_cast<const void *>(&ff_finish_kernel_multi), q_, grid_, block_, smem_,
                     kPdlKrylov);
        return;
    }
    pdl_launch(kPdlKrylov, &ff_finish_kernel, grid_, block_, smem_, s_, Hm, ldh, sv, k, Z, ld, x, x2, scale, n, first);
}

// a = b = hi + lo of the pairs, rounded once to FP64 (within 2^-53 of the
// pair's value); b may be null
__device__ __forceinline__ void ff_join_kernel_impl(int bid_, int nb_, const float2 *__restrict__ x2,
                                                    double *__restrict__ a, double *__restrict__ b, size_t n) {
    const size_t i = size_t(bid_) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float2 v = x2[i];
    const double r = join(v);
    a[i] = r;
    if (b) b[i] = r;
}
__global__ void ff_join_kernel(const float2 *__restrict__ x2, double *__restrict__ a, double *__restrict__ b,
                               size_t n) {
    pdl_wait();
    ff_join_kernel_impl(blockIdx.x, gridDim.x, x2, a, b, n);
}
struct ff_join_kernel_args {
    int nb_;
    const float2 *x2;
    double *a;
    double *b;
    size_t n;
};
__global__ void ff_join_kernel_multi(const __grid_constant__ MultiP<ff_join_kernel_args> M) {
    pdl_wait();
    int b_;
    const ff_join_kernel_args &q_ = M.a[merge_find(M.start, M.n, b_)];
    ff_join_kernel_impl(b_, q_.nb_, q_.x2, q_.a, q_.b, q_.n);
}
void ff_join_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, const float2 *x2, double *a,
                       double *b, size_t n) {
    if (Recorder *r_ = batch_recorder()) {
        ff_join_kernel_args q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.x2 = x2;
        q_.a = a;
        q_.b = b;
        q_.n = n;
        batch_record(r_, reinterpret_cast<const void *>(&ff_join_kernel_multi), q_, grid_, block_, smem_, kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &ff_join_kernel, grid_, block_, smem_, s_, x2, a, b, n);
}


// r = b - S x with x given split; S split in the packed FP64 layout (element
// j of facet e in 16-byte group (j / 2, e), lane j % 2, here two float pairs)

// res = b - S x in two-float arithmetic (x as split pairs), one thread per
// facet row: a block takes tiles of kResFacets facets in turn, thread (r, f) row r of
// facet f of the tile.  Bound by HBM (S as pairs, 40 (p+1)^2 bytes per facet): a thread
// issues the loads of its row first, then stages the pairs of its facet and of the four
// neighbours in shared memory (thread (r, f) component r of the five), then adds the
// 5 (p+1) products of its row in the order of the packed layout.  With one tile per
// block and the row's loads behind the staging, a tile cost a block the latency of four
// dependent loads and of the norm's handover: 52 instead of 70 us on 491,520 facets at
// p = 2 (200 MB, 3.8 TB/s), 36 instead of 41 on 196,608 at p = 3, 14.4 instead of 17.4 on
// 30,000 at p = 4.
// res may be null, and c32 names the FP32 start of an inner solve on res
// (F32Copy).  With partial non-null also ||res||^2: block sums of the rows'
// squares, the last block adding the block sums in block order into out[0]
// and handing the value to the host through pub (the value, a system fence,
// then seq).
constexpr int kResFacets = kResFFFacets;
template <int P> constexpr int kResPerSM = P == 1 ? 8 : P == 2 ? 5 : P == 3 ? 3 : 2;   // blocks per SM

// a load that stays where it is written (before the barrier of the staging)
__device__ __forceinline__ float4 load_now(const float4 *p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

template <int P>
__device__ __forceinline__ void residual_ff_kernel_impl(int bid_, int nb_, int NF, const float4 *__restrict__ S2,
                                                        const int32_t *__restrict__ nbr, const double *__restrict__ b,
                                                        const float2 *__restrict__ x2, double *__restrict__ res,
                                                        double *partial, unsigned int *counter, double *out,
                                                        HostValue *pub, int32_t seq, const F32Copy c32) {
    constexpr int PP = P + 1, RS = 5 * PP, NQR = (RS + 1) / 2;   // entries of a row, 16-byte groups it touches
    __shared__ float2 sx[5][PP][kResFacets];
    const int r = threadIdx.x / kResFacets, f = threadIdx.x % kResFacets;
    double sq = 0.0;
    for (int tile = bid_; tile * kResFacets < NF; tile += nb_) {
        const int e = tile * kResFacets + f;
        const bool on = e < NF;
        // row r holds entries j0 .. j0 + RS - 1, in groups q0 .. q0 + NQR - 1
        // (j0 is even whenever RS is, and the entry of lane g of group q0 + t
        // is then 2t + g of the row)
        const int j0 = r * RS, q0 = j0 / 2, odd = (RS % 2) ? (j0 & 1) : 0;
        float4 v[NQR];
        float2 xv[5];
        double bv = 0.0;
        if (on) {
#pragma unroll
            for (int t = 0; t < NQR; ++t) v[t] = load_now(S2 + size_t(q0 + t) * NF + e);
            bv = b[size_t(r) * NF + e];
            xv[0] = x2[size_t(r) * NF + e];
#pragma unroll
            for (int q = 1; q < 5; ++q) xv[q] = x2[size_t(r) * NF + __ldg(nbr + size_t(q - 1) * NF + e)];
        }
        if (tile != bid_) __syncthreads();     // the last tile's pairs have been read
        if (on) {
#pragma unroll
            for (int q = 0; q < 5; ++q) sx[q][r][f] = xv[q];
        }
        __syncthreads();
        if (!on) continue;
        FFAcc acc;
#pragma unroll
        for (int t = 0; t < NQR; ++t) {
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const int k = 2 * t + g - odd;
                if (k >= 0 && k < RS)
                    acc.add(g ? make_float2(v[t].z, v[t].w) : make_float2(v[t].x, v[t].y), sx[k / PP][k % PP][f]);
            }
        }
        const double rv = bv - acc.value();
        if (res) res[size_t(r) * NF + e] = rv;
        if (c32.b32) {
            c32.b32[size_t(r) * NF + e] = to_float(mul_pow2(rv, c32.scale));
            c32.z32[size_t(r) * NF + e] = 0.0f;
        }
        sq = fma(rv, rv, sq);
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
__global__ void __launch_bounds__(kResFacets * (P + 1), kResPerSM<P>) residual_ff_kernel(int NF, const float4 *__restrict__ S2,
                                                          const int32_t *__restrict__ nbr,
                                                          const double *__restrict__ b, const float2 *__restrict__ x2,
                                                          double *__restrict__ res, double *partial,
                                                          unsigned int *counter, double *out, HostValue *pub,
                                                          int32_t seq, const F32Copy c32) {
    pdl_wait();
    residual_ff_kernel_impl<P>(blockIdx.x, gridDim.x, NF, S2, nbr, b, x2, res, partial, counter, out, pub, seq, c32);
}
template <int P>
struct residual_ff_kernel_args {
    int nb_;
    int NF;
    const float4 *S2;
    const int32_t *nbr;
    const double *b;
    const float2 *x2;
    double *res;
    double *partial;
    unsigned int *counter;
    double *out;
    HostValue *pub;
    int32_t seq;
    F32Copy c32;
};
template <int P>
__global__ void __launch_bounds__(kResFacets * (P + 1), kResPerSM<P>) residual_ff_kernel_multi(const __grid_constant__ MultiP<residual_ff_kernel_args<P>> M) {
    pdl_wait();
    int b_;
    const residual_ff_kernel_args<P> &q_ = M.a[merge_find(M.start, M.n, b_)];
    residual_ff_kernel_impl<P>(b_, q_.nb_, q_.NF, q_.S2, q_.nbr, q_.b, q_.x2, q_.res, q_.partial, q_.counter, q_.out,
                               q_.pub, q_.seq, q_.c32);
}
template <int P>
void residual_ff_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int NF, const float4 *S2,
                           const int32_t *nbr, const double *b, const float2 *x2, double *res, double *partial,
                           unsigned int *counter, double *out, HostValue *pub, int32_t seq, const F32Copy &c32) {
    if (Recorder *r_ = batch_recorder()) {
        residual_ff_kernel_args<P> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.NF = NF;
        q_.S2 = S2;
        q_.nbr = nbr;
        q_.b = b;
        q_.x2 = x2;
        q_.res = res;
        q_.partial = partial;
        q_.counter = counter;
        q_.out = out;
        q_.pub = pub;
        q_.seq = seq;
        q_.c32 = c32;
        batch_record(r_, reinterpret_cast<const void *>(&residual_ff_kernel_multi<P>), q_, grid_, block_, smem_,
                     kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &residual_ff_kernel<P>, grid_, block_, smem_, s_, NF, S2, nbr, b, x2, res, partial, counter,
               out, pub, seq, c32);
}


// (r_u, r_h may live in page-locked host memory read over the C2C link; with
// cu, ch non-null each value read is also stored there, in HBM)
template <int NP>
__device__ __forceinline__ void stage_cell_rhs(int N, int K0, const double *__restrict__ r_u,
                                               const double *__restrict__ r_h, float2 (*sIn)[kCellsPad],
                                               double *__restrict__ cu = nullptr, double *__restrict__ ch = nullptr) {
    const int nc = min(kCells, N - K0);
    for (int j = threadIdx.x; j < nc * 2 * NP; j += blockDim.x) {
        const size_t k = size_t(K0) * 2 * NP + j;
        const double v = r_u[k];
        if (cu) cu[k] = v;
        sIn[j % (2 * NP)][j / (2 * NP)] = split(v);
    }
    for (int j = threadIdx.x; j < nc * NP; j += blockDim.x) {
        const size_t k = size_t(K0) * NP + j;
        const double v = r_h[k];
        if (ch) ch[k] = v;
        sIn[2 * NP + j % NP][j / NP] = split(v);
    }
}

// ---------------------------------------------------------------- the cell solve
// q = A_K^-1 M_K v for 32 cells per block (lane = cell), v in function space: the h rows
// of the stored R_M = A_K^-1 M_K, then the velocity from the momentum equations,
//   h = (R_M v)_h,   u = R (v_u - tau g G h),
// with the weak gradient G by reference matrices shared by all cells in the cell's J^-T,
// and R two n_p x n_p matrices (P, Q) or, where f is constant on every cell (FC), two
// numbers.  A cell reads 3 n_p^2 pairs (FC) or 5 n_p^2 instead of the 9 n_p^2 of R_M,
// with about as many products.  Only h is taken from a stored inverse on purpose:
// eliminating the velocity in two-float arithmetic as well (S^-1 (v_h - tau H div R v_u),
// n_p^2 pairs) reads less still, but the cancellation in that sum is amplified twice by
// the derivatives: 1.8e-12 instead of 1e-14 relative at p = 3, Courant 8.
// The warps take the rows in turn (kSolveWarps divides n_p).  sV holds v as pairs on
// entry and q on return (rows u_x, u_y, h; [33]: no bank conflicts); ends with a barrier.
template <int P> constexpr int kSolveWarps = P == 1 ? 3 : P == 2 ? 6 : 5;

__device__ __forceinline__ float2 ff_pair(const FFAcc &a) {
    const float hi = __fadd_rn(a.s, a.c);
    return make_float2(hi, __fsub_rn(a.c, __fsub_rn(hi, a.s)));
}
__device__ __forceinline__ float2 ff_neg(const float2 a) { return make_float2(-a.x, -a.y); }

struct SolveMat {
    const float4 *Hr2, *PQ2;    // tiles of the condensation
    const float2 *lgeo;
    const float4 *tab;          // FFTabOffsets
};

template <int P, bool FC>
__device__ __forceinline__ void cell_solve(const SolveMat &m, int tile, bool on, const float4 *tab,
                                           float2 (*sV)[kCellsPad]) {
    constexpr int NP = (P + 1) * (P + 2) / 2, NK = 3 * NP, CP = (NP + 1) / 2, KP = (NK + 1) / 2;
    constexpr int NW = kSolveWarps<P>, RW = NP / NW;
    constexpr FFTabOffsets O = ff_tab_offsets(P);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float2 *geo = m.lgeo + size_t(tile) * kLGeo * kCells + lane;
    const float4 *Hr = m.Hr2 + size_t(tile) * NP * KP * kCells + lane;
    const float4 *PQ = FC ? nullptr : m.PQ2 + size_t(tile) * 2 * NP * CP * kCells + lane;
    // padding cells of the last tile have no matrices: their lanes keep zeros
    float2 hv[RW];
#pragma unroll
    for (int u = 0; u < RW; ++u) {
        FFAcc acc;
        if (on) row_pairs<NK>(acc, Hr + size_t(w + u * NW) * KP * kCells, sV, lane);
        hv[u] = ff_pair(acc);
    }
    __syncthreads();                            // every warp has read v
#pragma unroll
    for (int u = 0; u < RW; ++u) sV[2 * NP + w + u * NW][lane] = hv[u];
    __syncthreads();
    // v_u - tau g G h
    if (on) {
        const float2 j00 = __ldg(geo), j01 = __ldg(geo + kCells), j10 = __ldg(geo + 2 * kCells),
                     j11 = __ldg(geo + 3 * kCells);
#pragma unroll
        for (int u = 0; u < RW; ++u) {
            const int i = w + u * NW;
            FFAcc g1, g2;
#pragma unroll 5
            for (int k = 0; k < NP; ++k) {
                const float4 d = tab[O.W + i * NP + k];
                const float2 h = sV[2 * NP + k][lane];
                g1.add(make_float2(d.x, d.y), h);
                g2.add(make_float2(d.z, d.w), h);
            }
            const float2 a1 = ff_neg(ff_pair(g1)), a2 = ff_neg(ff_pair(g2));
            const float2 vx = sV[i][lane], vy = sV[NP + i][lane];
            FFAcc x, y;
            x.s = vx.x;
            x.c = vx.y;
            x.add(j00, a1);
            x.add(j01, a2);
            y.s = vy.x;
            y.c = vy.y;
            y.add(j10, a1);
            y.add(j11, a2);
            float2 px = ff_pair(x), py = ff_pair(y);
            if constexpr (FC) {
                const float2 kap = __ldg(geo + 13 * kCells), fk = __ldg(geo + 14 * kCells);
                FFAcc ax, ay;
                ax.add(kap, px);
                ax.add(fk, py);
                ay.add(kap, py);
                ay.add(ff_neg(fk), px);
                px = ff_pair(ax);
                py = ff_pair(ay);
            }
            sV[i][lane] = px;
            sV[NP + i][lane] = py;
        }
    }
    __syncthreads();
    if constexpr (!FC) {
        // u = R (...): rows P x + Q y and P y - Q x
        float2 ux[RW], uy[RW];
#pragma unroll
        for (int u = 0; u < RW; ++u) {
            const int i = w + u * NW;
            FFAcc ax, ay;
            if (on) {
#pragma unroll 2
                for (int cp = 0; cp < CP; ++cp) {
                    const float4 p = __ldg(PQ + size_t(i * CP + cp) * kCells);
                    const float4 q = __ldg(PQ + size_t((NP + i) * CP + cp) * kCells);
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        const int k = 2 * cp + g;
                        if (k >= NP) break;
                        const float2 pk = g ? make_float2(p.z, p.w) : make_float2(p.x, p.y);
                        const float2 qk = g ? make_float2(q.z, q.w) : make_float2(q.x, q.y);
                        const float2 x = sV[k][lane], y = sV[NP + k][lane];
                        ax.add(pk, x);
                        ax.add(qk, y);
                        ay.add(pk, y);
                        ay.add(ff_neg(qk), x);
                    }
                }
            }
            ux[u] = ff_pair(ax);
            uy[u] = ff_pair(ay);
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < RW; ++u) {
            sV[w + u * NW][lane] = ux[u];
            sV[NP + w + u * NW][lane] = uy[u];
        }
        __syncthreads();
    }
}

// the cell solve's tables into shared memory (no barrier)
template <int P>
__device__ __forceinline__ void stage_tab(float4 *tab, const float4 *src) {
    for (int k = threadIdx.x; k < ff_tab_offsets(P).total; k += blockDim.x) tab[k] = __ldg(src + k);
}

// Step 1: z_K = A_K^-1 M_K r_K by the cell solve, stored as normalised pairs (z2
// [NK][N], when given) for step 3, and the cell rows ycell = C_K z_K: on edge i the
// flux H t_y u_x - H t_x u_y + tau_s |e| h at its p + 1 cell nodes, times the edge mass
// matrix.  Bound by HBM and FP32 issue together: 90 us on 131,072 cells at p = 3 with f
// constant per cell (430 MB, 4.8 TB/s), 123 us on 327,680 at p = 2 with f varying,
// against 186 and 176 us with the rows of the stored A_K^-1 M_K (1,029 MB, HBM-bound).
template <int P, bool FC>
__device__ __forceinline__ void rhs_cell_z_kernel_impl(int bid_, int nb_, int N, const SolveMat &m,
                                                       const double *__restrict__ r_u,
                                                       const double *__restrict__ r_h, double *__restrict__ ycell,
                                                       float2 *__restrict__ z2, double *__restrict__ cu,
                                                       double *__restrict__ ch) {
    constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2, NK = 3 * NP, M = 3 * PP, NW = kSolveWarps<P>;
    constexpr FFTabOffsets O = ff_tab_offsets(P);
    __shared__ float2 sV[NK][kCellsPad];
    __shared__ float2 sC[M][kCellsPad];        // edge fluxes
    __shared__ float4 tab[O.total];
    const int K0 = bid_ * kCells, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    stage_tab<P>(tab, m.tab);
    stage_cell_rhs<NP>(N, K0, r_u, r_h, sV, cu, ch);
    const int K = K0 + lane;
    const bool on = K < N;
    if (!on)
        for (int q = w; q < NK; q += NW) sV[q][lane] = make_float2(0.f, 0.f);
    __syncthreads();
    cell_solve<P, FC>(m, bid_, on, tab, sV);
    if (z2 && on)
        for (int q = w; q < NK; q += NW) z2[size_t(q) * N + K] = sV[q][lane];
    const float2 *geo = m.lgeo + size_t(bid_) * kLGeo * kCells + lane;
    for (int t = w; t < M; t += NW) {
        const int i = t / PP, b = edge_cell_node(P, i, t % PP);
        FFAcc acc;
        if (on) {
            acc.add(__ldg(geo + (4 + 3 * i) * kCells), sV[b][lane]);
            acc.add(__ldg(geo + (5 + 3 * i) * kCells), sV[NP + b][lane]);
            acc.add(__ldg(geo + (6 + 3 * i) * kCells), sV[2 * NP + b][lane]);
        }
        sC[t][lane] = ff_pair(acc);
    }
    __syncthreads();
    if (!on) return;
    for (int t = w; t < M; t += NW) {
        const int i = t / PP, jj = t % PP;
        FFAcc acc;
#pragma unroll
        for (int jb = 0; jb < PP; ++jb) {
            const float4 v = tab[O.m1 + jb * PP + jj];
            acc.add(make_float2(v.x, v.y), sC[i * PP + jb][lane]);
        }
        ycell[size_t(t) * N + K] = acc.value();
    }
}
template <int P, bool FC>
__global__ void __launch_bounds__(32 * kSolveWarps<P>) rhs_cell_z_kernel(int N, const SolveMat m,
                                                         const double *__restrict__ r_u,
                                                         const double *__restrict__ r_h, double *__restrict__ ycell,
                                                         float2 *__restrict__ z2, double *__restrict__ cu,
                                                         double *__restrict__ ch) {
    pdl_wait();
    rhs_cell_z_kernel_impl<P, FC>(blockIdx.x, gridDim.x, N, m, r_u, r_h, ycell, z2, cu, ch);
}
template <int P, bool FC>
struct rhs_cell_z_kernel_args {
    int nb_;
    int N;
    SolveMat m;
    const double *r_u;
    const double *r_h;
    double *ycell;
    float2 *z2;
    double *cu;
    double *ch;
};
template <int P, bool FC>
__global__ void __launch_bounds__(32 * kSolveWarps<P>) rhs_cell_z_kernel_multi(const __grid_constant__ MultiP<rhs_cell_z_kernel_args<P, FC>> M) {
    pdl_wait();
    int b_;
    const rhs_cell_z_kernel_args<P, FC> &q_ = M.a[merge_find(M.start, M.n, b_)];
    rhs_cell_z_kernel_impl<P, FC>(b_, q_.nb_, q_.N, q_.m, q_.r_u, q_.r_h, q_.ycell, q_.z2, q_.cu, q_.ch);
}
template <int P, bool FC>
void rhs_cell_z_kernel_go(unsigned grid_, unsigned block_, size_t smem_, cudaStream_t s_, int N, const SolveMat &m,
                          const double *r_u, const double *r_h, double *ycell, float2 *z2, double *cu, double *ch) {
    if (Recorder *r_ = batch_recorder()) {
        rhs_cell_z_kernel_args<P, FC> q_;
        std::memset(static_cast<void *>(&q_), 0, sizeof(q_));
        q_.nb_ = int(grid_);
        q_.N = N;
        q_.m = m;
        q_.r_u = r_u;
        q_.r_h = r_h;
        q_.ycell = ycell;
        q_.z2 = z2;
        q_.cu = cu;
        q_.ch = ch;
        batch_record(r_, reinterpret_cast<const void *>(&rhs_cell_z_kernel_multi<P, FC>), q_, grid_, block_, smem_,
                     kPdlFamily);
        return;
    }
    pdl_launch(kPdlFamily, &rhs_cell_z_kernel<P, FC>, grid_, block_, smem_, s_, N, m, r_u, r_h, ycell, z2, cu, ch);
}

// lambda on the block's cells (the pairs of its three facets' nodes in the cell's order)
template <int P>
__device__ __forceinline__ void stage_cell_trace(int N, int NF, int K0, const double *__restrict__ lam,
                                                 const int32_t *__restrict__ facet_of,
                                                 const int32_t *__restrict__ flip, float2 (*sL)[kCellsPad]) {
    constexpr int PP = P + 1, M = 3 * PP;
    const int nc = min(kCells, N - K0);
    for (int j = threadIdx.x; j < nc * M; j += blockDim.x) {
        const int cell = j / M, q = j % M, i = q / PP, jj = q % PP, K = K0 + cell;
        const int f = facet_of[3 * K + i], fl = flip[3 * K + i];
        sL[q][cell] = split(lam[size_t(fl ? P - jj : jj) * NF + f]);
    }
}

// Step 3 from explicit right-hand sides: q_K = A_K^-1 M_K r_K - X_B lambda_K, the cell
// solve of r and the stored X_B, written in the caller's u / h layout
template <int P, bool FC>
__global__ void __launch_bounds__(32 * kSolveWarps<P>) recover_ff_kernel(int N, int NF, const SolveMat m,
                                                         const float4 *__restrict__ Xb2, const double *__restrict__ r_u,
                                                         const double *__restrict__ r_h, const double *__restrict__ lam,
                                                         const int32_t *__restrict__ facet_of,
                                                         const int32_t *__restrict__ flip, double *__restrict__ u,
                                                         double *__restrict__ hout) {
    constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2, NK = 3 * NP, M = 3 * PP, NW = kSolveWarps<P>;
    constexpr int MP = (M + 1) / 2;
    constexpr FFTabOffsets O = ff_tab_offsets(P);
    __shared__ float2 sV[NK][kCellsPad];
    __shared__ float2 sL[M][kCellsPad];         // lambda on the cell's three facets
    __shared__ float4 tab[O.total];
    const int K0 = blockIdx.x * kCells, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nc = min(kCells, N - K0);
    stage_tab<P>(tab, m.tab);
    stage_cell_rhs<NP>(N, K0, r_u, r_h, sV);
    stage_cell_trace<P>(N, NF, K0, lam, facet_of, flip, sL);
    const bool on = K0 + lane < N;
    if (!on)
        for (int q = w; q < NK; q += NW) sV[q][lane] = make_float2(0.f, 0.f);
    __syncthreads();
    cell_solve<P, FC>(m, blockIdx.x, on, tab, sV);
    if (on) {
        for (int rho = w; rho < NK; rho += NW) {
            FFAcc acc;
            const float2 z = sV[rho][lane];
            acc.s = z.x;
            acc.c = z.y;
            row_pairs<M>(acc, Xb2 + (size_t(blockIdx.x) * NK * MP + size_t(rho) * MP) * kCells + lane, sL, lane, true);
            sV[rho][lane] = ff_pair(acc);
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < nc * 2 * NP; j += blockDim.x) {
        const float2 v = sV[j % (2 * NP)][j / (2 * NP)];
        u[size_t(K0) * 2 * NP + j] = join(v);
    }
    for (int j = threadIdx.x; j < nc * NP; j += blockDim.x) {
        const float2 v = sV[2 * NP + j % NP][j / NP];
        hout[size_t(K0) * NP + j] = join(v);
    }
}

// step 3 from the kept z_K: q_K = z_K - X_B lambda_K (two-float, z as the
// starting sum), written in the caller's u / h layout
template <int P>
__global__ void __launch_bounds__(256) recover_z_kernel(int N, int NF, const float2 *__restrict__ z2,
                                                        const float4 *__restrict__ Xb2,
                                                        const double *__restrict__ lam,
                                                        const int32_t *__restrict__ facet_of,
                                                        const int32_t *__restrict__ flip, double *__restrict__ u,
                                                        double *__restrict__ hout) {
    constexpr int PP = P + 1, NP = (P + 1) * (P + 2) / 2, NK = 3 * NP, M = 3 * PP, NW = 8;
    constexpr int MP = (M + 1) / 2;
    __shared__ float2 sIn[M][kCellsPad];        // lambda on the cell's three facets
    __shared__ double sOut[NK][kCellsPad];
    const int K0 = blockIdx.x * kCells, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nc = min(kCells, N - K0);
    stage_cell_trace<P>(N, NF, K0, lam, facet_of, flip, sIn);
    __syncthreads();
    const int K = K0 + lane;
    if (K < N) {
        for (int rho = w; rho < NK; rho += NW) {
            FFAcc acc;
            const float2 z = z2[size_t(rho) * N + K];
            acc.s = z.x;
            acc.c = z.y;
            row_pairs<M>(acc, Xb2 + (size_t(blockIdx.x) * NK * MP + size_t(rho) * MP) * kCells + lane, sIn, lane,
                         true);
            sOut[rho][lane] = acc.value();
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < nc * 2 * NP; j += blockDim.x)
        u[size_t(K0) * 2 * NP + j] = sOut[j % (2 * NP)][j / (2 * NP)];
    for (int j = threadIdx.x; j < nc * NP; j += blockDim.x) hout[size_t(K0) * NP + j] = sOut[2 * NP + j % NP][j / NP];
}

}  // namespace

cudaError_t launch_split(const double *a, float2 *out, size_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (n % 2) return cudaErrorInvalidValue;
    split_kernel<<<blocks(n / 2, 512), 256, 0, s>>>(reinterpret_cast<const double2 *>(a), reinterpret_cast<float4 *>(out),
                                                    n / 2);
    return cudaGetLastError();
}

cudaError_t launch_ff_axpy(float2 *x2, const float *d, const double *scale, size_t n, bool first, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    ff_axpy_kernel_go(blocks(n, 256), 256, 0, s, x2, d, scale, n, first ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_ff_finish(const double *Hm, int ldh, const double *sv, int k, const float *Z, size_t ld,
                             const float *x, float2 *x2, const double *scale, size_t n, bool first, cudaStream_t s) {
    if (n == 0 || k <= 0) return cudaSuccess;
    if (k > 64) return cudaErrorInvalidValue;
    const size_t per = size_t(256) * kFinU;
    ff_finish_kernel_go(unsigned((n + per - 1) / per), 256, sizeof(double) * size_t(k) * k, s, Hm, ldh, sv, k, Z, ld,
                        x, x2, scale, n, first ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_ff_join(const float2 *x2, double *a, double *b, size_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    ff_join_kernel_go(blocks(n, 256), 256, 0, s, x2, a, b, n);
    return cudaGetLastError();
}

cudaError_t launch_residual_ff(hdg_handle *h, const double *b, const float2 *x2, double *res, double *partial,
                               unsigned int *counter, double *out, HostValue *pub, int32_t seq, const F32Copy &c32) {
    // at most the blocks that 152 SMs hold, with about the same number of tiles each
    const unsigned tiles = blocks(h->NF, kResFacets);
    HDG_DISPATCH_P(h->p, (residual_ff_kernel_go<P>(blocks(tiles, int(blocks(tiles, 152 * kResPerSM<P>))),
                                                   kResFacets * (P + 1), 0, h->stream, h->NF,
                                                   reinterpret_cast<const float4 *>(h->d_Sval2), h->d_nbr, b, x2, res,
                                                   partial, counter, out, pub, seq, c32)));
    return cudaGetLastError();
}

namespace {
SolveMat solve_mat(const hdg_handle *h) {
    return SolveMat{reinterpret_cast<const float4 *>(h->d_Hr2), reinterpret_cast<const float4 *>(h->d_PQ2), h->d_lgeo,
                    h->d_fftab};
}
}  // namespace

cudaError_t launch_rhs_z(hdg_handle *h, const double *r_u, const double *r_h, double *g, double *ycell, float2 *z2,
                         double *copy_u, double *copy_h, const NormOut &nrm) {
    const SolveMat m = solve_mat(h);
    const unsigned nb = blocks(h->N, kCells);
    if (h->f_const) {
        HDG_DISPATCH_P(h->p, (rhs_cell_z_kernel_go<P, true>(nb, 32 * kSolveWarps<P>, 0, h->stream, h->N, m, r_u, r_h,
                                                            ycell, z2, copy_u, copy_h)));
    } else {
        HDG_DISPATCH_P(h->p, (rhs_cell_z_kernel_go<P, false>(nb, 32 * kSolveWarps<P>, 0, h->stream, h->N, m, r_u, r_h,
                                                             ycell, z2, copy_u, copy_h)));
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_rhs_gather(h, ycell, g, nrm);
}

cudaError_t launch_recover_z(hdg_handle *h, const float2 *z2, const double *lam, double *u, double *hout) {
    HDG_DISPATCH_P(h->p, (recover_z_kernel<P><<<blocks(h->N, kCells), 256, 0, h->stream>>>(
                             h->N, h->NF, z2, reinterpret_cast<const float4 *>(h->d_Xb2), lam, h->d_facet_of,
                             h->d_flip, u, hout)));
    return cudaGetLastError();
}

cudaError_t launch_recover_ff(hdg_handle *h, const double *r_u, const double *r_h, const double *lam, double *u,
                              double *hout) {
    const SolveMat m = solve_mat(h);
    const unsigned nb = blocks(h->N, kCells);
    if (h->f_const) {
        HDG_DISPATCH_P(h->p, (recover_ff_kernel<P, true><<<nb, 32 * kSolveWarps<P>, 0, h->stream>>>(
                                 h->N, h->NF, m, reinterpret_cast<const float4 *>(h->d_Xb2), r_u, r_h, lam,
                                 h->d_facet_of, h->d_flip, u, hout)));
    } else {
        HDG_DISPATCH_P(h->p, (recover_ff_kernel<P, false><<<nb, 32 * kSolveWarps<P>, 0, h->stream>>>(
                                 h->N, h->NF, m, reinterpret_cast<const float4 *>(h->d_Xb2), r_u, r_h, lam,
                                 h->d_facet_of, h->d_flip, u, hout)));
    }
    return cudaGetLastError();
}

}  // namespace hdg
