// Device and host helpers shared by the sparse kernels of the inner loop (kernels_sparse.cu,
// kernels_inner.cu): row loads, deterministic block / grid reductions, the float-pair slack
// diagonal, ELL fetches, and the last-block bookkeeping of the SpMM and the line search.
#pragma once

#include <cmath>
#include <mutex>
#include <unordered_map>

#include "dev_util.cuh"
#include "fpair.cuh"
#include "quartic.cuh"

namespace alm {

template <typename T>
__device__ __forceinline__ typename VecT<T>::type load_row(const T *__restrict__ R, int64_t i, int ldr, int gl,
                                                           bool active) {
    constexpr int W = VecT<T>::W;
    return active ? ldro(R + i * ldr + gl * W) : vzero(T());
}

// Block sums of v[0..NV) (NV <= 8) into out[0..NV), valid in thread 0.  The values share the
// butterfly: in each of its first rounds a lane keeps half of its values and hands over the
// other half, so that eight values take 9 FP64 additions a warp instead of 40 (an FP64
// instruction holds a warp 64 cycles, and the kernel waits for these sums at its end).  shm holds
// (warps of the block) x 8 doubles.
template <int NV>
__device__ __forceinline__ void block_sums(const double (&v)[NV], double (&out)[NV], double *shm) {
    constexpr int K = NV <= 1 ? 1 : NV <= 2 ? 2 : NV <= 4 ? 4 : 8;
    static_assert(NV <= 8, "at most eight values");
    double a[K];
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] = k < NV ? v[k] : 0.0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int idx = 0;
#pragma unroll
    for (int h = K / 2, o = 16; h > 0; h >>= 1, o >>= 1) {
        const bool up = lane & o;
        idx += up ? h : 0;
#pragma unroll
        for (int u = 0; u < h; ++u) {
            const double give = up ? a[u] : a[u + h], keep = up ? a[u + h] : a[u];
            a[u] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
#pragma unroll
    for (int o = 16 / K; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    __syncthreads();  // shm may still be read from the sums before
    if ((lane & (32 / K - 1)) == 0) shm[warp * 8 + idx] = a[0];
    __syncthreads();
    if (warp == 0) {
        double t = 0.0;
        if (lane < NV)
            for (int w = 0; w < int(blockDim.x >> 5); ++w) t += shm[w * 8 + lane];
#pragma unroll
        for (int k = 0; k < NV; ++k) out[k] = __shfl_sync(0xffffffffu, t, k);
    }
}

// In the last block: deterministic sums over blocks of the partial slots 0..NV-1, all
// slots loaded in one pass (results valid in thread 0).
template <int NV>
__device__ __forceinline__ void sum_partials_n(const double *partials, double (&out)[NV], double *shm) {
    double t[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) t[k] = out[k] = 0.0;
    for (int b = threadIdx.x; b < int(gridDim.x); b += blockDim.x)
#pragma unroll
        for (int k = 0; k < NV; ++k) t[k] += __ldcg(partials + size_t(b) * kPartStride + k);
    block_sums<NV>(t, out, shm);
}

// write the block sums of vals[0..NV) to part[0..NV)
template <int NV>
__device__ __forceinline__ void block_partials(const double (&vals)[NV], double *part, double *shm) {
    double out[NV];
    block_sums<NV>(vals, out, shm);
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) part[k] = out[k];
}

// a double as a float pair hi + lo (FP32 form) or as itself (FP64 form)
template <typename T>
__device__ __forceinline__ void store_slack_diag(const SparseView<T> &v, int64_t i, double d) {
    T hi, lo;
    split_pair(d, hi, lo);
    v.d_s[i] = hi;
    if (v.d_s_lo) v.d_s_lo[i] = lo;
}

// ---------------------------------------------------------------------------------------
// inner-loop slack update for diagonal-selector problems (MaxCut): with y fixed during an
// inner solve, S_ii = (C_ii - a_i y_k) + sigma a_i (a_i |r_i|^2 - b_k) = base_i + sigma a_i res_i.
// base_i is a float pair computed once per outer iteration; res_i is formed from the
// compensated |r_i|^2 in float-pair arithmetic (the subtraction of b_k ~ 1 is where FP32
// would lose the residual), so the whole update runs in FP32 on one streaming pass over R.
// ---------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void slack_pair(const SparseView<T> &v, int64_t i, T xh, T xl, T sigma, T &dh_out,
                                           T &dl_out) {
    const int k = v.d_sel_k[i];
    T dh = v.base_hi[i], dl = v.base_lo ? v.base_lo[i] : T(0);
    if (k >= 0) {
        const T a = sizeof(T) == 8 ? T(v.d_sel_a[i]) : T(v.d_sel_af[i]);
        const T ph = a * xh;
        const T pe = fma(a, xh, -ph) + a * xl;
        const T s0 = ph - v.b_hi[i];
        const T bb = s0 - ph;
        const T e0 = (ph - (s0 - bb)) + (-v.b_hi[i] - bb);
        const T res = s0 + (e0 + pe - (v.b_lo ? v.b_lo[i] : T(0)));
        const T corr = sigma * a * res;
        const T s1 = dh + corr;
        const T b1 = s1 - dh;
        dl += (dh - (s1 - b1)) + (corr - b1);
        dh = s1;
    }
    dh_out = dh;
    dl_out = dl;
}

// ---------------------------------------------------------------------------------------
// ELL forms of the SpMM and of the line-search SDDMM (static S_off, rows of at most KF
// entries).  One row per group and iteration; the column indices and values of the
// group's next row are fetched before the current row's gathers are issued, so that a
// row costs one memory latency instead of a chain of three.
// ---------------------------------------------------------------------------------------
template <typename T, int KF>
__device__ __forceinline__ void ell_fetch(const int *__restrict__ cols, const T *__restrict__ vals, int64_t row,
                                          int (&jj)[KF], T (&ss)[KF]) {
    const int4 *cp = reinterpret_cast<const int4 *>(cols + row * KF);
#pragma unroll
    for (int q = 0; q < KF / 4; ++q) {
        const int4 c = __ldg(cp + q);
        jj[4 * q] = c.x;
        jj[4 * q + 1] = c.y;
        jj[4 * q + 2] = c.z;
        jj[4 * q + 3] = c.w;
    }
#pragma unroll
    for (int k = 0; k < KF; ++k) ss[k] = __ldg(vals + row * KF + k);
}
template <typename T, int K>
__device__ __forceinline__ void ell_fetch2(const int *__restrict__ cols, const T *__restrict__ vals, int64_t row,
                                           int (&jj)[K], T (&ss)[K]) {  // K = 2 (8-byte rows)
    const int2 c = __ldg(reinterpret_cast<const int2 *>(cols + row * K));
    jj[0] = c.x;
    jj[1] = c.y;
    ss[0] = __ldg(vals + row * K);
    ss[1] = __ldg(vals + row * K + 1);
}

// last-block bookkeeping of the inner CG step (shared by the CSR and ELL SpMMs)
__device__ __forceinline__ void spmm_finish(DevState *st, double gg, double go, double gd, double zg) {
    st->gg = gg;
    if (!isfinite(gg)) {
        st->status = ALM_ERR_NUMERIC;
        st->done = 1;
    } else if (sqrt(gg) <= st->tau_abs) {
        st->done = 1;
    }
    double beta = 0.0;
    if (!st->restart && st->method == ALM_INNER_CG && st->zg_prev > 0.0) {
        beta = fmax(0.0, (zg - go) / st->zg_prev);
        if (-zg + beta * gd >= 0.0) beta = 0.0;  // not a descent direction: restart
    }
    st->beta = beta;
    st->g_gprev = go;
    st->g_dprev = gd;
    st->gg_prev = gg;
    st->zg = zg;
    st->zg_prev = zg;
    st->restart = 0;
}

// thread 0 of the last block of a line-search SDDMM: FP64 quartic coefficients, the
// exact step and (MODE 1) the inner-loop bookkeeping
template <typename T, int MODE, bool LR>
__device__ __forceinline__ void ls_finish(const SparseView<T> &v, DevState *st, int r, const double (&tot)[5]) {
        double s1 = tot[0], s2 = tot[1];
        const double a11 = tot[2], a12 = tot[3], a22 = tot[4];
        if (LR)  // <s u u^T, RD^T + DR^T> = 2 s (R^T u).(D^T u),  <s u u^T, DD^T> = s |D^T u|^2
            for (int l = 0; l < v.lr_k; ++l) {
                double zr = 0.0, dd = 0.0;
                for (int col = 0; col < r; ++col) {
                    zr += st->z[l][col] * st->zd[l][col];
                    dd += st->zd[l][col] * st->zd[l][col];
                }
                s1 += v.lr_s[l] * 2.0 * zr;
                s2 += v.lr_s[l] * dd;
            }
        const double sigma = st->sigma;
        double q[5];
        // MODE 1: q0 has no part in the step, and L is not computed in the inner loop (st->L is some
        // earlier call's); at a restart beta = 0 and <G, D_old> is of whatever D_old holds.  Neither may
        // reach the test for non-finite coefficients below.
        q[0] = MODE == 1 ? 0.0 : st->L;
        if (MODE == 1) q[1] = -st->zg + (st->beta != 0.0 ? st->beta * st->g_dprev : 0.0);  // <G, D>, D = -Z + beta D_old
        else q[1] = s1;
        q[2] = s2 + 0.5 * sigma * a11;
        q[3] = sigma * a12;
        q[4] = 0.5 * sigma * a22;
        st->c1 = s1;
        st->c2 = s2;
        st->a11 = a11;
        st->a12 = a12;
        st->a22 = a22;
        for (int k = 0; k < 5; ++k) st->q[k] = q[k];
        int unb = 0;
        const double alpha = quartic_argmin(q, &unb);
        st->alpha = unb ? 0.0 : alpha;
        if (MODE == 1) {
            bool finite = true;
            for (int k = 0; k < 5; ++k) finite = finite && isfinite(q[k]);
            if (!finite) {
                st->status = ALM_ERR_NUMERIC;
                st->done = 1;
            } else if (unb) {
                st->status = ALM_ERR_UNBOUNDED;
                st->done = 1;
            } else if (!(alpha > 0.0)) {
                st->done = 1;
            } else {
                st->iters += 1;
                if (st->iters >= st->max_inner) st->done = 2;
            }
        } else if (unb) {
            st->status = ALM_ERR_UNBOUNDED;
            st->alpha = INFINITY;
        }
    }

// the line search's scalars to the host
__device__ __forceinline__ void ls_result(HostResult *res, const DevState *st) {
    for (int k = 0; k < 5; ++k) res->q[k] = st->q[k];
    res->alpha = st->alpha;
    res->status = st->status;
    __threadfence_system();
}

// blocks of kBlock threads per SM that the kernel can keep resident (cached per kernel)
static int resident_blocks(const void *fn) {
    static std::mutex mu;
    static std::unordered_map<const void *, int> cache;
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(fn);
    if (it != cache.end()) return it->second;
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, kBlock, 0) != cudaSuccess || b < 1) {
        (void)cudaGetLastError();
        b = 1;
    }
    cache[fn] = b;
    return b;
}

template <typename K>
static int grid_for(const LaunchCtx &c, K *fn, int64_t items, int64_t items_per_block) {
    int64_t need = (items + items_per_block - 1) / items_per_block;
    if (need < 1) need = 1;
    int64_t cap = int64_t(c.sms) * resident_blocks(reinterpret_cast<const void *>(fn));
    if (cap > c.grid) cap = c.grid;
    return int(need < cap ? need : cap);
}

static inline int lanes_for(int r, int W) {
    const int nvec = (r + W - 1) / W;
    int L = 1;
    while (L < nvec) L <<= 1;
    return L;
}

#define ALM_DISPATCH_LANES(L, ...)                                \
    switch (L) {                                                  \
        case 1: { constexpr int LN = 1; __VA_ARGS__; } break;    \
        case 2: { constexpr int LN = 2; __VA_ARGS__; } break;    \
        case 4: { constexpr int LN = 4; __VA_ARGS__; } break;    \
        case 8: { constexpr int LN = 8; __VA_ARGS__; } break;    \
        default: { constexpr int LN = 16; __VA_ARGS__; } break;  \
    }

}  // namespace alm
