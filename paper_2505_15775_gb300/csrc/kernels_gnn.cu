// Warm-start network: forward, loss and backward kernels (inference and training).
//
// The network predicts (R0, y0) for a unit-diagonal SDP from C alone (motivation: the
// local convergence of ALM-BM in Sec. 4.2 needs a starting factor near a solution and a
// multiplier near y*).  Three message-passing layers of width 64 on the pattern of C,
//     agg_i = (sum_j a_ij h_j) / max(deg_i, 1),   h'_i = relu(Ws h_i + Wn agg_i + b),
// a_ij = C_ij / mean|C_ij|, then the heads rhat_i = W_R h_i (32 columns) and
// yhat_i = w_y . h_i + b_y.  Activations are stored in BF16 (or FP32) and every product
// accumulates in FP32; gradients are FP32.  The products are FP32 FMAs in a fixed order per
// output, so that a row's activations have the same bits in every tile size and batch (accuracy
// does not ask for it: the error against 64 bits is BF16 storage's, 2.5e-3 on the warm start of
// the torus; FP32 weights in BF16 parts on the tensor cores have not been tried).  A 64-wide
// layer is then 8192 FMAs a row, bound by the FP32 pipe, provided that its operands come from
// registers: tiles of rows (k_gnn_layer), each thread 8 rows x 4 outputs.
//
// Rows are the global rows of a batch (alm_batch); row g belongs to instance
// row_inst[g], whose first row is row_off[row_inst[g]] and whose pattern uses local
// column indices.
#include <cuda_bf16.h>

#include <cmath>

#include "dev_util.cuh"
#include "gnn_internal.h"

namespace alm {
namespace {

__device__ __forceinline__ float tof(float x) { return x; }
__device__ __forceinline__ float tof(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T>
__device__ __forceinline__ T fromf(float x);
template <>
__device__ __forceinline__ float fromf<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 fromf<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

__device__ __forceinline__ float warp_sumf(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// SplitMix64 counter generator mapped to [-1, 1) (the same definition as the Lanczos
// start vector)
// (m 2^-52 - 1 for the 53-bit integer m, which FP64 holds exactly, rounded to float once:
// the integer m - 2^52 converted and scaled gives the same float without the FP64 pipe)
__device__ __forceinline__ float smx_pm1(uint64_t seed, uint64_t i) {
    uint64_t z = seed + (i + 1) * 0x9e3779b97f4a7c15ULL;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    z ^= z >> 31;
    return __ll2float_rn(static_cast<long long>(z >> 11) - (1LL << 52)) * 0x1p-52f;
}

// x_i = [1, deg_i/dbar, s_i/sbar, log(n)/8, u_1..u_4]
template <typename T>
__global__ void k_gnn_features(GnnGraph g, uint64_t feat_seed, T *__restrict__ H0) {
    for (int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < g.rows; r += int64_t(gridDim.x) * blockDim.x) {
        const int b = g.row_inst[r];
        const float4 sc = g.scal[b];
        const int e0 = g.rowptr[r], e1 = g.rowptr[r + 1];
        float s = 0.f;
        for (int e = e0; e < e1; ++e) s += g.val[e];
        const uint64_t li = uint64_t(r - g.row_off[b]);
        T *h = H0 + r * kGnnFeat;
        h[0] = fromf<T>(1.f);
        h[1] = fromf<T>(float(e1 - e0) * sc.x);
        h[2] = fromf<T>(s * sc.z);
        h[3] = fromf<T>(sc.w);
        for (int k = 0; k < 4; ++k) h[4 + k] = fromf<T>(smx_pm1(feat_seed + uint64_t(k), li));
    }
}

// two neighbouring channels of a row
__device__ __forceinline__ float2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ float2 ld2(const __nv_bfloat16 *p) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
}
// ... as loaded, for loads that are to be in flight together: a conversion behind a condition makes the
// compiler wait for each
__device__ __forceinline__ float2 ld2_raw(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ unsigned ld2_raw(const __nv_bfloat16 *p) { return *reinterpret_cast<const unsigned *>(p); }
__device__ __forceinline__ float2 to_f2(float2 x) { return x; }
__device__ __forceinline__ float2 to_f2(unsigned x) { return __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&x)); }
__device__ __forceinline__ void st2(float *p, float x, float y) { *reinterpret_cast<float2 *>(p) = make_float2(x, y); }
__device__ __forceinline__ void st2(__nv_bfloat16 *p, __nv_bfloat16 x, __nv_bfloat16 y) {
    *reinterpret_cast<__nv_bfloat162 *>(p) = __halves2bfloat162(x, y);
}
// four neighbouring channels
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16 *p) {
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st4(float *p, const float (&q)[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(q[0], q[1], q[2], q[3]);
}
__device__ __forceinline__ void st4(__nv_bfloat16 *p, const float (&q)[4]) {
    st2(p, __float2bfloat16_rn(q[0]), __float2bfloat16_rn(q[1]));
    st2(p + 2, __float2bfloat16_rn(q[2]), __float2bfloat16_rn(q[3]));
}
// N consecutive floats of shared memory (N = 2 or a multiple of 4) into registers
template <int N>
__device__ __forceinline__ void lds_vec(const float *p, float (&x)[N]) {
    if constexpr (N == 2) {
        const float2 v = *reinterpret_cast<const float2 *>(p);
        x[0] = v.x;
        x[1] = v.y;
    } else {
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const float4 v = *reinterpret_cast<const float4 *>(p + 4 * q);
            x[4 * q] = v.x;
            x[4 * q + 1] = v.y;
            x[4 * q + 2] = v.z;
            x[4 * q + 3] = v.w;
        }
    }
}

// One layer over tiles of TR rows: agg_i, h'_i = relu(Ws h_i + Wn agg_i + b), and with HEADS
// (the last layer) rhat_i = W_R h'_i, yhat_i = w_y . h'_i + b_y from the tile in shared memory.
// STORE: keep agg and, in the last layer, h' for the backward pass (inference needs neither).
//   gather   64 channels: a warp loads the places of all its rows and their first 32 entries at
//            once (a lane per row, then a lane per entry: the dependent loads are paid once a
//            tile), then takes four rows at a time, a lane two channels of each, with the gathers
//            of sixteen neighbour rows in flight; what a row has beyond 64 entries is gathered by
//            itself, sixteen at a time (warm start on a graph with hubs of 30,000 entries, BF16:
//            15.0 -> 8.5 ms; Kronecker of 2^14 rows 1.54 -> 0.54 ms).  8 channels: two threads a row.
//   product  thread (rg, og) holds TR / 16 rows x 4 outputs; inputs lie transposed in shared
//            memory ([channel][row]), so an input costs TR / 16 x 4 FMAs per 16-byte load.
//            Per output the FMAs run over k in order, Wn's before Ws's, from the bias on.
// 128 rows a tile hold the FP32 pipe busy (6 shared loads per 64 FMAs); fewer rows than one
// such tile per multiprocessor take tiles of 32, to use more of them.  us of alm_gnn_warm_start,
// tiles of 32 / 128, ER graphs of degree 10, BF16 (FP32): 8,000 rows 90 / 113 (90 / 106), 16,000
// 119 / 118 (120 / 110), 19,456 (the line) 119 / 117 (120 / 108), 32,000 158 / 131 (153 / 129).
// Bound: the FP32 pipe (8192 FMAs a row: 0.21 ms per million rows) and the gathers.  One warp
// per row with both operands of every FMA from shared memory took 1.25 ms a layer on 1e6 torus
// rows and 0.37 ms for the heads: alm_gnn_warm_start 3.60 -> 1.50 ms.
template <int DIN, int TR, bool HEADS>
constexpr int gnn_layer_smem() {
    return 4 * (DIN * (2 * kGnnHid + 4) + kGnnHid + 2 * DIN * (TR + 4) +
                (HEADS ? kGnnHid * (kGnnRank + 4) + kGnnHid : 0));
}
template <typename T, int DIN, int TR, bool HEADS, bool STORE>
__global__ void __launch_bounds__(256, 2) k_gnn_layer(GnnGraph g, GnnLayerArgs<T> p) {
    extern __shared__ __align__(16) float gsm[];
    constexpr int WP = 2 * kGnnHid + 4;  // pitch of [k][Ws row | Wn row]
    constexpr int TP = TR + 4;           // pitch of [k][row]
    constexpr int RPT = TR / 16;         // rows per thread of the product
    float *w = gsm, *bs = w + DIN * WP, *hx = bs + kGnnHid, *ax = hx + DIN * TP, *wr = ax + DIN * TP;
    float *wy = wr + kGnnHid * (kGnnRank + 4);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int t = tid; t < kGnnHid * DIN; t += 256) {
        const int o = t / DIN, k = t % DIN;
        w[k * WP + o] = p.Ws[t];
        w[k * WP + kGnnHid + o] = p.Wn[t];
    }
    for (int t = tid; t < kGnnHid; t += 256) bs[t] = p.bias[t];
    float by = 0.f;
    if (HEADS) {
        for (int t = tid; t < kGnnRank * kGnnHid; t += 256) wr[(t % kGnnHid) * (kGnnRank + 4) + t / kGnnHid] = p.WR[t];
        for (int t = tid; t < kGnnHid; t += 256) wy[t] = p.wy[t];
        by = p.by[0];
    }
    __syncthreads();
    const int og = tid & 15, rg = tid >> 4;
    for (int64_t r0 = int64_t(blockIdx.x) * TR; r0 < g.rows; r0 += int64_t(gridDim.x) * TR) {
        if constexpr (DIN == kGnnHid) {
            constexpr int RW = TR / 8;  // rows of a warp: their places and first 32 entries in one go
            int64_t base = 0;
            int e0 = 0, dg = 0;
            float icb = 0.f;
            if (lane < RW && r0 + wid * RW + lane < g.rows) {
                const int64_t r = r0 + wid * RW + lane;
                const int b = g.row_inst[r];
                base = g.row_off[b];
                icb = g.scal[b].y;
                e0 = g.rowptr[r];
                dg = g.rowptr[r + 1] - e0;
            }
            int jc[RW];
            float ac[RW];
#pragma unroll
            for (int q = 0; q < RW; ++q) {
                const int eq = __shfl_sync(0xffffffffu, e0, q), dq = __shfl_sync(0xffffffffu, dg, q);
                const float iq = __shfl_sync(0xffffffffu, icb, q);
                jc[q] = lane < dq ? g.col[eq + lane] : 0;
                ac[q] = lane < dq ? g.val[eq + lane] * iq : 0.f;
            }
#pragma unroll
            for (int q4 = 0; q4 < RW; q4 += 4) {  // four rows at once
                const int lr = wid * RW + q4;
                float a0[4] = {0.f, 0.f, 0.f, 0.f}, a1[4] = {0.f, 0.f, 0.f, 0.f};
                int deg[4];
                const T *hb[4];
                int most = 0;
                float2 own[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    deg[q] = __shfl_sync(0xffffffffu, dg, q4 + q);
                    most = max(most, deg[q]);
                    hb[q] = p.H + __shfl_sync(0xffffffffu, base, q4 + q) * DIN + 2 * lane;
                    const int64_t r = r0 + lr + q;
                    own[q] = r < g.rows ? ld2(p.H + r * DIN + 2 * lane) : make_float2(0.f, 0.f);
                }
                for (int c0 = 0; c0 < min(most, 64); c0 += 32) {  // 32 entries of each row at a time
                    int jr[4];
                    float aw[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        jr[q] = jc[q4 + q];
                        aw[q] = ac[q4 + q];
                        if (c0 > 0) {
                            const int eq = __shfl_sync(0xffffffffu, e0, q4 + q) + c0 + lane;
                            const float iq = __shfl_sync(0xffffffffu, icb, q4 + q);
                            const bool in = c0 + lane < deg[q];
                            jr[q] = in ? g.col[eq] : 0;
                            aw[q] = in ? g.val[eq] * iq : 0.f;
                        }
                    }
                    const int lim = min(32, most - c0);
                    for (int t = 0; t < lim; t += 4) {
                        float2 x[4][4];
                        float a[4][4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int j = __shfl_sync(0xffffffffu, jr[q], t + u);
                                a[u][q] = __shfl_sync(0xffffffffu, aw[q], t + u);
                                x[u][q] = make_float2(0.f, 0.f);
                                if (c0 + t + u < deg[q]) x[u][q] = ld2(hb[q] + int64_t(j) * DIN);
                            }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                if (c0 + t + u < deg[q]) {  // warp-uniform
                                    a0[q] = fmaf(a[u][q], x[u][q].x, a0[q]);
                                    a1[q] = fmaf(a[u][q], x[u][q].y, a1[q]);
                                }
                    }
                }
                // the rest of longer rows, one row at a time with sixteen of its entries in flight and the
                // next 32 places on their way (a hub among three short rows had four)
                if (most > 64)
#pragma unroll 1
                    for (int q = 0; q < 4; ++q) {
                        const int dq = __shfl_sync(0xffffffffu, dg, q4 + q);
                        if (dq <= 64) continue;
                        const int eq = __shfl_sync(0xffffffffu, e0, q4 + q);
                        const float iq = __shfl_sync(0xffffffffu, icb, q4 + q);
                        const T *hq = p.H + __shfl_sync(0xffffffffu, base, q4 + q) * DIN + 2 * lane;
                        float s0 = q == 0 ? a0[0] : q == 1 ? a0[1] : q == 2 ? a0[2] : a0[3];
                        float s1 = q == 0 ? a1[0] : q == 1 ? a1[1] : q == 2 ? a1[2] : a1[3];
                        int jn = 64 + lane < dq ? g.col[eq + 64 + lane] : 0;
                        float an = 64 + lane < dq ? g.val[eq + 64 + lane] * iq : 0.f;
                        for (int c0 = 64; c0 < dq; c0 += 32) {
                            const int jr = jn, left = min(32, dq - c0);
                            const float aw = an;
                            const bool more = c0 + 32 + lane < dq;
                            jn = more ? g.col[eq + c0 + 32 + lane] : 0;
                            an = more ? g.val[eq + c0 + 32 + lane] * iq : 0.f;
                            for (int t = 0; t < left; t += 16) {
                                decltype(ld2_raw(hq)) raw[16];
#pragma unroll
                                for (int u = 0; u < 16; ++u)  // past the row: column 0, not used
                                    raw[u] = ld2_raw(hq + int64_t(__shfl_sync(0xffffffffu, jr, t + u)) * DIN);
#pragma unroll
                                for (int u = 0; u < 16; ++u) {
                                    const float a = __shfl_sync(0xffffffffu, aw, t + u);
                                    const float2 x = to_f2(raw[u]);
                                    if (t + u < left) {
                                        s0 = fmaf(a, x.x, s0);
                                        s1 = fmaf(a, x.y, s1);
                                    }
                                }
                            }
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (k == q) {
                                a0[k] = s0;
                                a1[k] = s1;
                            }
                    }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float inv = 1.f / float(max(deg[q], 1));
                    const T q0 = fromf<T>(a0[q] * inv), q1 = fromf<T>(a1[q] * inv);
                    if (STORE && r0 + lr + q < g.rows) st2(p.AGG + (r0 + lr + q) * DIN + 2 * lane, q0, q1);
                    a0[q] = tof(q0);  // the backward sees the stored (rounded) value
                    a1[q] = tof(q1);
                }
                *reinterpret_cast<float4 *>(hx + (2 * lane) * TP + lr) = make_float4(own[0].x, own[1].x, own[2].x, own[3].x);
                *reinterpret_cast<float4 *>(hx + (2 * lane + 1) * TP + lr) = make_float4(own[0].y, own[1].y, own[2].y, own[3].y);
                *reinterpret_cast<float4 *>(ax + (2 * lane) * TP + lr) = make_float4(a0[0], a0[1], a0[2], a0[3]);
                *reinterpret_cast<float4 *>(ax + (2 * lane + 1) * TP + lr) = make_float4(a1[0], a1[1], a1[2], a1[3]);
            }
        } else {
            for (int t = tid; t < 2 * TR; t += 256) {  // two threads a row, four channels each
                const int lr = t >> 1, c = 4 * (t & 1);
                const int64_t r = r0 + lr;
                float q[4] = {0.f, 0.f, 0.f, 0.f}, h[4] = {0.f, 0.f, 0.f, 0.f};
                if (r < g.rows) {
                    const int b = g.row_inst[r];
                    const int64_t base = g.row_off[b];
                    const float icb = g.scal[b].y;
                    const int e0 = g.rowptr[r], deg = g.rowptr[r + 1] - e0;
                    const float4 o = ld4(p.H + r * DIN + c);
                    h[0] = o.x, h[1] = o.y, h[2] = o.z, h[3] = o.w;
                    constexpr int U = TR == 32 ? 8 : 4;  // in flight; 64 threads gather for a tile of 32 rows
                    for (int t = 0; t < deg; t += U) {  // by offset: e0 + t may be near 2^31
                        float4 x[U];
                        float a[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int ee = e0 + min(t + u, deg - 1);
                            a[u] = g.val[ee] * icb;
                            x[u] = ld4(p.H + (base + g.col[ee]) * DIN + c);
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (t + u < deg) {
                                q[0] = fmaf(a[u], x[u].x, q[0]);
                                q[1] = fmaf(a[u], x[u].y, q[1]);
                                q[2] = fmaf(a[u], x[u].z, q[2]);
                                q[3] = fmaf(a[u], x[u].w, q[3]);
                            }
                    }
                    const float inv = 1.f / float(max(deg, 1));
#pragma unroll
                    for (int k = 0; k < 4; ++k) q[k] = tof(fromf<T>(q[k] * inv));
                    if (STORE) st4(p.AGG + r * DIN + c, q);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    hx[(c + k) * TP + lr] = h[k];
                    ax[(c + k) * TP + lr] = q[k];
                }
            }
        }
        __syncthreads();
        float z[RPT][4];
#pragma unroll
        for (int i = 0; i < RPT; ++i)
#pragma unroll
            for (int o = 0; o < 4; ++o) z[i][o] = bs[4 * og + o];
#pragma unroll 4
        for (int k = 0; k < DIN; ++k) {
            float h[RPT], a[RPT], ws[4], wn[4];
            lds_vec<RPT>(hx + k * TP + RPT * rg, h);
            lds_vec<RPT>(ax + k * TP + RPT * rg, a);
            lds_vec<4>(w + k * WP + 4 * og, ws);
            lds_vec<4>(w + k * WP + kGnnHid + 4 * og, wn);
#pragma unroll
            for (int i = 0; i < RPT; ++i)
#pragma unroll
                for (int o = 0; o < 4; ++o) z[i][o] = fmaf(ws[o], h[i], fmaf(wn[o], a[i], z[i][o]));
        }
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int64_t r = r0 + RPT * rg + i;
#pragma unroll
            for (int o = 0; o < 4; ++o) z[i][o] = tof(fromf<T>(fmaxf(z[i][o], 0.f)));
            if ((!HEADS || STORE) && r < g.rows) st4(p.Hout + r * kGnnHid + 4 * og, z[i]);
        }
        __syncthreads();  // hx and ax may be overwritten
        if constexpr (HEADS) {
#pragma unroll
            for (int o = 0; o < 4; ++o)
#pragma unroll
                for (int i = 0; i < RPT; ++i) hx[(4 * og + o) * TP + RPT * rg + i] = z[i][o];
            __syncthreads();
            constexpr int RPH = TR / 32;  // rows per thread of the factor head (8 threads a row)
            const int cg = tid & 7, rh = (tid >> 3) * RPH;
            float acc[RPH][4];
#pragma unroll
            for (int i = 0; i < RPH; ++i)
#pragma unroll
                for (int o = 0; o < 4; ++o) acc[i][o] = 0.f;
#pragma unroll 4
            for (int k = 0; k < kGnnHid; ++k) {
                float v[4];
                lds_vec<4>(wr + k * (kGnnRank + 4) + 4 * cg, v);
#pragma unroll
                for (int i = 0; i < RPH; ++i) {
                    const float h = hx[k * TP + rh + i];
#pragma unroll
                    for (int o = 0; o < 4; ++o) acc[i][o] = fmaf(v[o], h, acc[i][o]);
                }
            }
#pragma unroll
            for (int i = 0; i < RPH; ++i)
                if (r0 + rh + i < g.rows)
                    *reinterpret_cast<float4 *>(p.rhat + (r0 + rh + i) * kGnnRank + 4 * cg) =
                        make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            for (int lr = tid; lr < TR; lr += 256)
                if (r0 + lr < g.rows) {
                    float t[kGnnHid / 2];  // pairs and then halves: 7 roundings deep, two chains would be 33
#pragma unroll
                    for (int k = 0; k < kGnnHid / 2; ++k)
                        t[k] = fmaf(wy[k], hx[k * TP + lr], wy[k + kGnnHid / 2] * hx[(k + kGnnHid / 2) * TP + lr]);
#pragma unroll
                    for (int o = kGnnHid / 4; o > 0; o >>= 1)
#pragma unroll
                        for (int k = 0; k < o; ++k) t[k] += t[k + o];
                    p.yhat[r0 + lr] = t[0] + by;
                }
            __syncthreads();
        }
    }
}

// R0 = normalise(rhat/|rhat| + mix u/|u|), u_i a seeded uniform row (SplitMix64 stream
// mix_seed, element 32 i + c): mixing keeps R0 of full rank when the network's rows span
// few directions.  A zero row becomes u/|u| (e_1 if mix = 0).  y0 = cbar * yhat.
// 8 lanes per row (float4).
__global__ void k_gnn_warm(GnnGraph g, const float *__restrict__ rhat, const float *__restrict__ yhat,
                           const double *__restrict__ cbar, float mix, uint64_t mix_seed, float *__restrict__ R0,
                           double *__restrict__ y0) {
    const int lane = threadIdx.x & 31, gl = lane & 7;
    const unsigned gm = 0xffu << (lane & ~7);
    const int64_t ng = (int64_t(gridDim.x) * blockDim.x) >> 3;
    for (int64_t r = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 3; r < g.rows; r += ng) {
        const float4 v = *reinterpret_cast<const float4 *>(rhat + r * kGnnRank + gl * 4);
        const uint64_t li = uint64_t(r - g.row_off[g.row_inst[r]]) * kGnnRank + gl * 4;
        const float4 u = make_float4(smx_pm1(mix_seed, li), smx_pm1(mix_seed, li + 1), smx_pm1(mix_seed, li + 2),
                                     smx_pm1(mix_seed, li + 3));
        float s = v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        float su = u.x * u.x + u.y * u.y + u.z * u.z + u.w * u.w;
        for (int o = 4; o > 0; o >>= 1) {
            s += __shfl_xor_sync(gm, s, o);
            su += __shfl_xor_sync(gm, su, o);
        }
        const float a = s > 0.f ? rsqrtf(s) : 0.f;
        const float bmix = su > 0.f ? mix * rsqrtf(su) : 0.f;
        float4 w = make_float4(a * v.x + bmix * u.x, a * v.y + bmix * u.y, a * v.z + bmix * u.z, a * v.w + bmix * u.w);
        float sw = w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
        for (int o = 4; o > 0; o >>= 1) sw += __shfl_xor_sync(gm, sw, o);
        float4 out;
        if (sw > 0.f) {
            const float inv = rsqrtf(sw);
            out = make_float4(w.x * inv, w.y * inv, w.z * inv, w.w * inv);
        } else {
            out = make_float4(gl == 0 ? 1.f : 0.f, 0.f, 0.f, 0.f);
        }
        *reinterpret_cast<float4 *>(R0 + r * kGnnRank + gl * 4) = out;
        if (gl == 0) y0[r] = cbar[g.row_inst[r]] * double(yhat[r]);
    }
}

// Loss and its gradient w.r.t. the heads' outputs, 8 lanes per row i (a float4 of columns each):
//   e_ii = |rhat_i|^2 - |r*_i|^2,  e_ij = rhat_i.rhat_j - r*_i.r*_j (j a pattern neighbour)
//   dL/drhat_i = (4/np) e_ii rhat_i + (2/np) sum_j e_ij rhat_j   (both (i,j) and (j,i) in the
//   full pattern, so each unordered pair reaches both rows);  loss terms e_ii^2 and, for j > i,
//   e_ij^2;  ey = yhat_i - y*_i/cbar,  dL/dyhat_i = 2 lam ey / nrow.
// One reduction (3 shuffles) of the difference per neighbour; bound by the gathers of two
// 128-byte rows per neighbour.  Per-block loss partials in part[block].
__device__ __forceinline__ float dot4(float4 a, float4 b) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, a.x * b.x)));
}
__device__ __forceinline__ float oct_sum(float x, unsigned m) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(m, x, o);
    return x;
}
__global__ void __launch_bounds__(256) k_gnn_loss(GnnGraph g, const float *__restrict__ rhat,
                                                  const float *__restrict__ yhat, const float *__restrict__ Rs,
                                                  const double *__restrict__ ys, const double *__restrict__ cbar,
                                                  float inv_np, float lam_nrow, int rs_vec, float *__restrict__ dR,
                                                  float *__restrict__ dY, double *__restrict__ part) {
    __shared__ double red[8];
    // the caller's rows may lie at any float address
    auto ldrs = [&](int64_t row, int c) {
        const float *q = Rs + row * kGnnRank + c;
        return rs_vec ? ld4(q) : make_float4(q[0], q[1], q[2], q[3]);
    };
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, gl = lane & 7;
    const unsigned gm = 0xffu << (lane & ~7);
    float lsum = 0.f, lcomp = 0.f;
    for (int64_t r = int64_t(blockIdx.x) * 32 + (threadIdx.x >> 3); r < g.rows; r += int64_t(gridDim.x) * 32) {
        const int b = g.row_inst[r];
        const int64_t base = g.row_off[b];
        const int64_t li = r - base;
        const float4 ri = ld4(rhat + r * kGnnRank + 4 * gl), si = ldrs(r, 4 * gl);
        const float eii = oct_sum(dot4(ri, ri) - dot4(si, si), gm);
        const float c0 = 4.f * inv_np * eii;
        float4 d = make_float4(c0 * ri.x, c0 * ri.y, c0 * ri.z, c0 * ri.w);
        float le = eii * eii;
        const int e0 = g.rowptr[r], deg = g.rowptr[r + 1] - e0;
        int n0 = 0 < deg ? g.col[e0] : 0, n1 = 1 < deg ? g.col[e0 + 1] : n0;
        for (int t = 0; t < deg; t += 2) {  // by offset: e0 + t may be near 2^31
            const bool two = t + 1 < deg;
            const int j0 = n0, j1 = two ? n1 : j0;
            n0 = t + 2 < deg ? g.col[e0 + t + 2] : 0;  // the next round's, ahead of this one's gathers
            n1 = t + 3 < deg ? g.col[e0 + t + 3] : n0;
            const float4 ra = ld4(rhat + (base + j0) * kGnnRank + 4 * gl), sa = ldrs(base + j0, 4 * gl);
            const float4 rb = ld4(rhat + (base + j1) * kGnnRank + 4 * gl), sb = ldrs(base + j1, 4 * gl);
            const float ea = oct_sum(dot4(ri, ra) - dot4(si, sa), gm);
            const float eb = two ? oct_sum(dot4(ri, rb) - dot4(si, sb), gm) : 0.f;  // uniform in the group
            const float ca = 2.f * inv_np * ea, cb = 2.f * inv_np * eb;
            d = make_float4(fmaf(cb, rb.x, fmaf(ca, ra.x, d.x)), fmaf(cb, rb.y, fmaf(ca, ra.y, d.y)),
                            fmaf(cb, rb.z, fmaf(ca, ra.z, d.z)), fmaf(cb, rb.w, fmaf(ca, ra.w, d.w)));
            if (j0 > li) le += ea * ea;
            if (j1 > li) le += eb * eb;
        }
        *reinterpret_cast<float4 *>(dR + r * kGnnRank + 4 * gl) = d;
        if (gl == 0) {
            const float ey = float(double(yhat[r]) - ys[r] / cbar[b]);
            dY[r] = 2.f * lam_nrow * ey;
            const float t = le * inv_np + lam_nrow * ey * ey;
            const float s2 = lsum + t;  // two-sum
            const float bb = s2 - lsum;
            lcomp += (lsum - (s2 - bb)) + (t - bb);
            lsum = s2;
        }
    }
    double l = double(lsum) + double(lcomp);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) red[wid] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

// The backward kernels work on tiles of kBwdRows rows in shared memory, 256 threads, two CTAs
// per multiprocessor, each CTA walking tiles with its weight-gradient outputs in registers
// (written once, as this block's vector of partials: part[block * ldp + parameter offset]).
// A product's operands come as 16-byte shared loads for tiles of 4 x 4 or 4 x 8 outputs a
// thread.  One warp per row with operands from shared memory, a kernel for each weight matrix
// and a serial sum of 304 partials for each took 2.7 ms for a gradient on 137,000 rows
// (1.1 M edges); the tiles take 1.2 ms, forward pass included.
constexpr int kBwdRows = 64;
constexpr int kBwdPitch = kGnnHid + 4;

// Heads: dW_R = dR^T H3, dw_y = dY^T H3, db_y = sum dY, and the last layer's
// dZ = (W_R^T dR + w_y dY) (.) [H3 > 0]
template <typename T>
__global__ void __launch_bounds__(256, 2) k_gnn_heads_bwd(int64_t rows, const float *__restrict__ dR,
                                                          const float *__restrict__ dY, const T *__restrict__ H,
                                                          const float *__restrict__ WR, const float *__restrict__ wy,
                                                          float *__restrict__ dZ, float *__restrict__ part, int64_t ldp,
                                                          int off_WR, int off_wy, int off_by) {
    __shared__ __align__(16) float dt[kGnnRank][kBwdRows + 4], hs[kBwdRows][kBwdPitch], wr[kGnnRank][kBwdPitch];
    __shared__ __align__(16) float drow[kBwdRows][kGnnRank + 4], wys[kGnnHid], dys[kBwdRows];
    const int tid = threadIdx.x;
    for (int t = tid; t < kGnnRank * kGnnHid; t += 256) wr[t / kGnnHid][t % kGnnHid] = WR[t];
    if (tid < kGnnHid) wys[tid] = wy[tid];
    const int kg = tid & 15, mg = tid >> 4;  // 4 channels x (2 columns | 4 rows)
    float acc[2][4], accy = 0.f, accb = 0.f;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[m][k] = 0.f;
    for (int64_t r0 = int64_t(blockIdx.x) * kBwdRows; r0 < rows; r0 += int64_t(gridDim.x) * kBwdRows) {
        __syncthreads();
        for (int t = tid; t < kBwdRows * (kGnnRank / 4); t += 256) {
            const int lr = t / (kGnnRank / 4), c = 4 * (t % (kGnnRank / 4));
            const float4 x = r0 + lr < rows ? ld4(dR + (r0 + lr) * kGnnRank + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            *reinterpret_cast<float4 *>(&drow[lr][c]) = x;
            dt[c][lr] = x.x, dt[c + 1][lr] = x.y, dt[c + 2][lr] = x.z, dt[c + 3][lr] = x.w;
        }
        for (int t = tid; t < kBwdRows * (kGnnHid / 4); t += 256) {
            const int lr = t / (kGnnHid / 4), c = 4 * (t % (kGnnHid / 4));
            *reinterpret_cast<float4 *>(&hs[lr][c]) =
                r0 + lr < rows ? ld4(H + (r0 + lr) * kGnnHid + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (tid < kBwdRows) dys[tid] = r0 + tid < rows ? dY[r0 + tid] : 0.f;
        __syncthreads();
#pragma unroll 4
        for (int lr = 0; lr < kBwdRows; ++lr) {
            float h[4], d[2];
            lds_vec<4>(&hs[lr][4 * kg], h);
            lds_vec<2>(&drow[lr][2 * mg], d);
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[m][k] = fmaf(d[m], h[k], acc[m][k]);
        }
        if (tid < kGnnHid) {
            for (int lr = 0; lr < kBwdRows; ++lr) accy = fmaf(dys[lr], hs[lr][tid], accy);
        } else if (tid == kGnnHid) {
            for (int lr = 0; lr < kBwdRows; ++lr) accb += dys[lr];
        }
        float z[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) z[i][k] = wys[4 * kg + k] * dys[4 * mg + i];
#pragma unroll 4
        for (int c = 0; c < kGnnRank; ++c) {
            float d[4], w[4];
            lds_vec<4>(&dt[c][4 * mg], d);
            lds_vec<4>(&wr[c][4 * kg], w);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k) z[i][k] = fmaf(w[k], d[i], z[i][k]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int lr = 4 * mg + i;
            if (r0 + lr >= rows) continue;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (!(hs[lr][4 * kg + k] > 0.f)) z[i][k] = 0.f;
            st4(dZ + (r0 + lr) * kGnnHid + 4 * kg, z[i]);
        }
    }
    float *p = part + int64_t(blockIdx.x) * ldp;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int k = 0; k < 4; ++k) p[off_WR + (2 * mg + m) * kGnnHid + 4 * kg + k] = acc[m][k];
    if (tid < kGnnHid) p[off_wy + tid] = accy;
    else if (tid == kGnnHid) p[off_by] = accb;
}

// One 64-wide layer: dWs = dZ^T H, dWn = dZ^T AGG, db = sum dZ, and of its input
// dHp = Ws^T dZ (the direct part) and U = (Wn^T dZ) / max(deg, 1) (its aggregation's adjoint is
// applied by k_gnn_agg_t)
template <typename T>
constexpr int gnn_bwd_smem() { return 4 * (4 * kBwdRows * kBwdPitch + 2 * kGnnHid * kGnnHid); }
template <typename T>
__global__ void __launch_bounds__(256, 2) k_gnn_layer_bwd(GnnGraph g, const float *__restrict__ Ws,
                                                          const float *__restrict__ Wn, const T *__restrict__ H,
                                                          const T *__restrict__ AGG, const float *__restrict__ dZ,
                                                          float *__restrict__ dHp, float *__restrict__ U,
                                                          float *__restrict__ part, int64_t ldp, int off_Ws, int off_Wn,
                                                          int off_b) {
    extern __shared__ __align__(16) float gsm[];
    constexpr int P = kBwdPitch;
    float *ws = gsm, *wn = ws + kGnnHid * kGnnHid, *dz = wn + kGnnHid * kGnnHid;  // dz: [row][o]
    float *dzt = dz + kBwdRows * P, *hs = dzt + kBwdRows * P, *as = hs + kBwdRows * P;  // dzt: [o][row]
    const int tid = threadIdx.x;
    for (int t = tid; t < kGnnHid * kGnnHid; t += 256) {
        ws[t] = Ws[t];
        wn[t] = Wn[t];
    }
    const int kg = tid & 15, mg = tid >> 4;
    float accs[4][4], accn[4][4], accb = 0.f;
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int k = 0; k < 4; ++k) accs[m][k] = accn[m][k] = 0.f;
    for (int64_t r0 = int64_t(blockIdx.x) * kBwdRows; r0 < g.rows; r0 += int64_t(gridDim.x) * kBwdRows) {
        __syncthreads();
        for (int t = tid; t < kBwdRows * (kGnnHid / 4); t += 256) {
            const int lr = t / (kGnnHid / 4), c = 4 * (t % (kGnnHid / 4));
            const int64_t r = r0 + lr;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 d = r < g.rows ? ld4(dZ + r * kGnnHid + c) : zero;
            *reinterpret_cast<float4 *>(dz + lr * P + c) = d;
            dzt[c * P + lr] = d.x, dzt[(c + 1) * P + lr] = d.y, dzt[(c + 2) * P + lr] = d.z, dzt[(c + 3) * P + lr] = d.w;
            *reinterpret_cast<float4 *>(hs + lr * P + c) = r < g.rows ? ld4(H + r * kGnnHid + c) : zero;
            *reinterpret_cast<float4 *>(as + lr * P + c) = r < g.rows ? ld4(AGG + r * kGnnHid + c) : zero;
        }
        __syncthreads();
#pragma unroll 2
        for (int lr = 0; lr < kBwdRows; ++lr) {
            float d[4], h[4], a[4];
            lds_vec<4>(dz + lr * P + 4 * mg, d);
            lds_vec<4>(hs + lr * P + 4 * kg, h);
            lds_vec<4>(as + lr * P + 4 * kg, a);
#pragma unroll
            for (int m = 0; m < 4; ++m)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    accs[m][k] = fmaf(d[m], h[k], accs[m][k]);
                    accn[m][k] = fmaf(d[m], a[k], accn[m][k]);
                }
        }
        if (tid < kGnnHid)
            for (int lr = 0; lr < kBwdRows; ++lr) accb += dz[lr * P + tid];
        float s[4][4], u[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) s[i][k] = u[i][k] = 0.f;
#pragma unroll 2
        for (int o = 0; o < kGnnHid; ++o) {
            float d[4], w[4], v[4];
            lds_vec<4>(dzt + o * P + 4 * mg, d);
            lds_vec<4>(ws + o * kGnnHid + 4 * kg, w);
            lds_vec<4>(wn + o * kGnnHid + 4 * kg, v);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    s[i][k] = fmaf(w[k], d[i], s[i][k]);
                    u[i][k] = fmaf(v[k], d[i], u[i][k]);
                }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t r = r0 + 4 * mg + i;
            if (r >= g.rows) continue;
            const float inv = 1.f / float(max(g.rowptr[r + 1] - g.rowptr[r], 1));
#pragma unroll
            for (int k = 0; k < 4; ++k) u[i][k] *= inv;
            st4(dHp + r * kGnnHid + 4 * kg, s[i]);
            st4(U + r * kGnnHid + 4 * kg, u[i]);
        }
    }
    float *p = part + int64_t(blockIdx.x) * ldp;
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            p[off_Ws + (4 * mg + m) * kGnnHid + 4 * kg + k] = accs[m][k];
            p[off_Wn + (4 * mg + m) * kGnnHid + 4 * kg + k] = accn[m][k];
        }
    if (tid < kGnnHid) p[off_b + tid] = accb;
}

// The first layer's weight gradients (its input has none): dWs = dZ^T H0, dWn = dZ^T AGG0, db
template <typename T>
__global__ void __launch_bounds__(256) k_gnn_first_bwd(int64_t rows, const T *__restrict__ H,
                                                       const T *__restrict__ AGG, const float *__restrict__ dZ,
                                                       float *__restrict__ part, int64_t ldp, int off_Ws, int off_Wn,
                                                       int off_b) {
    __shared__ __align__(16) float dz[kBwdRows][kBwdPitch], xs[kBwdRows][2 * kGnnFeat + 4];
    const int tid = threadIdx.x, kk = tid & 15, mg = tid >> 4;  // input kk (H0 | AGG0), outputs 4 mg ..
    float acc[4] = {0.f, 0.f, 0.f, 0.f}, accb = 0.f;
    for (int64_t r0 = int64_t(blockIdx.x) * kBwdRows; r0 < rows; r0 += int64_t(gridDim.x) * kBwdRows) {
        __syncthreads();
        for (int t = tid; t < kBwdRows * (kGnnHid / 4); t += 256) {
            const int lr = t / (kGnnHid / 4), c = 4 * (t % (kGnnHid / 4));
            *reinterpret_cast<float4 *>(&dz[lr][c]) =
                r0 + lr < rows ? ld4(dZ + (r0 + lr) * kGnnHid + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        {
            const int lr = tid >> 2, c = 4 * (tid & 1);
            const T *src = (tid & 2) ? AGG : H;
            *reinterpret_cast<float4 *>(&xs[lr][((tid & 2) ? kGnnFeat : 0) + c]) =
                r0 + lr < rows ? ld4(src + (r0 + lr) * kGnnFeat + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
#pragma unroll 4
        for (int lr = 0; lr < kBwdRows; ++lr) {
            float d[4];
            lds_vec<4>(&dz[lr][4 * mg], d);
            const float x = xs[lr][kk];
#pragma unroll
            for (int m = 0; m < 4; ++m) acc[m] = fmaf(d[m], x, acc[m]);
        }
        if (tid < kGnnHid)
            for (int lr = 0; lr < kBwdRows; ++lr) accb += dz[lr][tid];
    }
    float *p = part + int64_t(blockIdx.x) * ldp + (kk < kGnnFeat ? off_Ws : off_Wn) + kk % kGnnFeat;
#pragma unroll
    for (int m = 0; m < 4; ++m) p[(4 * mg + m) * kGnnFeat] = acc[m];
    if (tid < kGnnHid) part[int64_t(blockIdx.x) * ldp + off_b + tid] = accb;
}

// The previous layer's dZ_i = (dHp_i + sum_{j in N(i)} a_ij U_j) (.) [H_i > 0] (the pattern is
// symmetric), one warp per row, a lane two channels; the row's columns and weights are loaded
// by the lanes beforehand, so that eight 256-byte gathers are in flight
template <typename T>
__global__ void __launch_bounds__(256, 5) k_gnn_agg_t(GnnGraph g, const float *__restrict__ U,
                                                   const float *__restrict__ dHp, const T *__restrict__ H,
                                                   float *__restrict__ dZ) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t nwarps = int64_t(gridDim.x) * 8;
    for (int64_t r = int64_t(blockIdx.x) * 8 + wid; r < g.rows; r += nwarps) {
        const int b = g.row_inst[r];
        const int64_t base = g.row_off[b];
        const float icb = g.scal[b].y;
        const int e0 = g.rowptr[r], deg = g.rowptr[r + 1] - e0;
        const float2 d = ld2(dHp + r * kGnnHid + 2 * lane), h = ld2(H + r * kGnnHid + 2 * lane);
        float s0 = 0.f, s1 = 0.f;
        const float *Ub = U + base * kGnnHid + 2 * lane;
        int jn = lane < deg ? g.col[e0 + lane] : 0;
        float an = lane < deg ? g.val[e0 + lane] * icb : 0.f;
        for (int c0 = 0; c0 < deg; c0 += 32) {
            const int jl = jn, lim = min(32, deg - c0);
            const float al = an;
            const bool more = c0 + 32 + lane < deg;
            jn = more ? g.col[e0 + c0 + 32 + lane] : 0;
            an = more ? g.val[e0 + c0 + 32 + lane] * icb : 0.f;
            for (int t = 0; t < lim; t += 8) {
                float2 x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int j = __shfl_sync(0xffffffffu, jl, t + u);
                    x[u] = t + u < lim ? ld2(Ub + int64_t(j) * kGnnHid) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {  // lanes past the row hold weight 0
                    const float a = __shfl_sync(0xffffffffu, al, t + u);
                    s0 = fmaf(a, x[u].x, s0);
                    s1 = fmaf(a, x[u].y, s1);
                }
            }
        }
        st2(dZ + r * kGnnHid + 2 * lane, h.x > 0.f ? d.x + s0 : 0.f, h.y > 0.f ? d.y + s1 : 0.f);
    }
}

// grad[k] = sum over blocks of part[b * ldp + k], k < cnt, and the loss, in a fixed order: 32
// parameters x 8 slices of the blocks per CTA, float pairs (an FP64 add holds a warp 64 cycles)
__global__ void __launch_bounds__(256) k_gnn_reduce(const float *__restrict__ part, int nblk, int64_t ldp, int cnt,
                                                    float *__restrict__ grad, const double *__restrict__ lpart,
                                                    int nl, double *__restrict__ loss) {
    __shared__ float hs[8][32], ls[8][32];
    __shared__ double red[8];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    if (int(blockIdx.x) == int(gridDim.x) - 1) {  // the last CTA: the loss
        double t = 0.0;
        for (int b = threadIdx.x; b < nl; b += 256) t += lpart[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (x == 0) red[y] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < 8; ++w) s += red[w];
            *loss = s;
        }
        return;
    }
    const int k = blockIdx.x * 32 + x;
    float h = 0.f, l = 0.f;
    auto add = [&](float v) {
        const float s = h + v;
        const float bb = s - h;
        l += (h - (s - bb)) + (v - bb);
        h = s;
    };
    if (k < cnt)
        for (int b = y; b < nblk; b += 8) add(part[int64_t(b) * ldp + k]);
    hs[y][x] = h;
    ls[y][x] = l;
    __syncthreads();
    if (y == 0 && k < cnt) {
        for (int w = 1; w < 8; ++w) {
            add(hs[w][x]);
            l += ls[w][x];
        }
        grad[k] = h + l;
    }
}

// Adam (Kingma and Ba, ICLR 2015) with bias correction
__global__ void k_gnn_adam(float *__restrict__ theta, const float *__restrict__ grad, float *__restrict__ m,
                           float *__restrict__ v, int cnt, float lr, float b1, float b2, float eps, float c1,
                           float c2) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
        const float g = grad[k];
        const float mk = b1 * m[k] + (1.f - b1) * g;
        const float vk = b2 * v[k] + (1.f - b2) * g * g;
        m[k] = mk;
        v[k] = vk;
        theta[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    }
}

}  // namespace

// ---------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------
static int warp_grid(int64_t rows, int sms) {
    const int64_t need = (rows + 7) / 8;
    const int64_t cap = int64_t(sms) * 8;
    return int(std::max<int64_t>(1, std::min(need, cap)));
}

template <typename T, int DIN, int TR, bool HEADS, bool STORE>
static cudaError_t layer_launch(const GnnGraph &g, const GnnLayerArgs<T> &p, int sms, cudaStream_t s) {
    auto *fn = k_gnn_layer<T, DIN, TR, HEADS, STORE>;
    constexpr int smem = gnn_layer_smem<DIN, TR, HEADS>();
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    const int64_t tiles = (g.rows + TR - 1) / TR;
    const int per = DIN == kGnnHid && TR == 128 ? 2 : 4;  // resident CTAs per multiprocessor
    fn<<<int(std::max<int64_t>(1, std::min<int64_t>(tiles, int64_t(sms) * per))), 256, smem, s>>>(g, p);
    return cudaGetLastError();
}

template <typename T, int TR, bool STORE>
static cudaError_t layers_launch(const GnnGraph &g, const GnnParams &p, GnnActs<T> &a, float *rhat, float *yhat,
                                 int sms, cudaStream_t s) {
    for (int l = 0; l < kGnnLayers; ++l) {
        const GnnLayerArgs<T> q{p.Ws[l], p.Wn[l], p.b[l], p.WR, p.wy, p.by, a.H[l], a.AGG[l], a.H[l + 1], rhat, yhat};
        const cudaError_t e = l == 0              ? layer_launch<T, kGnnFeat, TR, false, STORE>(g, q, sms, s)
                              : l + 1 < kGnnLayers ? layer_launch<T, kGnnHid, TR, false, STORE>(g, q, sms, s)
                                                   : layer_launch<T, kGnnHid, TR, true, STORE>(g, q, sms, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t gnn_forward(const GnnGraph &g, const GnnParams &p, uint64_t feat_seed, GnnActs<T> &a, float *rhat,
                        float *yhat, bool store, int sms, cudaStream_t s) {
    k_gnn_features<T><<<std::max<int64_t>(1, std::min<int64_t>((g.rows + 255) / 256, int64_t(sms) * 8)), 256, 0, s>>>(
        g, feat_seed, a.H[0]);
    if (g.rows >= int64_t(128) * sms)
        return store ? layers_launch<T, 128, true>(g, p, a, rhat, yhat, sms, s)
                     : layers_launch<T, 128, false>(g, p, a, rhat, yhat, sms, s);
    return store ? layers_launch<T, 32, true>(g, p, a, rhat, yhat, sms, s)
                 : layers_launch<T, 32, false>(g, p, a, rhat, yhat, sms, s);
}

cudaError_t gnn_warm(const GnnGraph &g, const float *rhat, const float *yhat, const double *cbar, float mix,
                     uint64_t mix_seed, float *R0, double *y0, int sms, cudaStream_t s) {
    const int64_t need = (g.rows * 8 + 255) / 256;
    k_gnn_warm<<<int(std::max<int64_t>(1, std::min<int64_t>(need, int64_t(sms) * 8))), 256, 0, s>>>(
        g, rhat, yhat, cbar, mix, mix_seed, R0, y0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t gnn_loss_grad(const GnnGraph &g, const GnnParams &p, float *grad, GnnActs<T> &a, const float *rhat,
                          const float *yhat, const float *Rs, const double *ys, const double *cbar, double lam,
                          double n_pattern, double n_rows, double *loss_dev, int sms, cudaStream_t s) {
    const GnnParams at = gnn_views(grad);
    auto off = [grad](const float *q) { return int(q - grad); };  // in the parameter vector
    const int lgrid = int(std::max<int64_t>(1, std::min<int64_t>((g.rows + 31) / 32, int64_t(sms) * 8)));
    k_gnn_loss<<<lgrid, 256, 0, s>>>(g, rhat, yhat, Rs, ys, cbar, float(1.0 / n_pattern), float(lam / n_rows),
                                     reinterpret_cast<uintptr_t>(Rs) % 16 == 0, a.dR, a.dY, a.lpart);
    const int nblk = int(std::min<int64_t>(a.nblk, (g.rows + kBwdRows - 1) / kBwdRows));
    k_gnn_heads_bwd<T><<<nblk, 256, 0, s>>>(g.rows, a.dR, a.dY, a.H[kGnnLayers], p.WR, p.wy, a.dZ, a.part, a.ldp,
                                            off(at.WR), off(at.wy), off(at.by));
    cudaError_t e = cudaFuncSetAttribute(k_gnn_layer_bwd<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         gnn_bwd_smem<T>());
    if (e != cudaSuccess) return e;
    for (int l = kGnnLayers - 1; l > 0; --l) {
        k_gnn_layer_bwd<T><<<nblk, 256, gnn_bwd_smem<T>(), s>>>(g, p.Ws[l], p.Wn[l], a.H[l], a.AGG[l], a.dZ, a.dHp,
                                                               a.U, a.part, a.ldp, off(at.Ws[l]), off(at.Wn[l]),
                                                               off(at.b[l]));
        k_gnn_agg_t<T><<<warp_grid(g.rows, sms), 256, 0, s>>>(g, a.U, a.dHp, a.H[l], a.dZ);
    }
    k_gnn_first_bwd<T><<<nblk, 256, 0, s>>>(g.rows, a.H[0], a.AGG[0], a.dZ, a.part, a.ldp, off(at.Ws[0]),
                                            off(at.Wn[0]), off(at.b[0]));
    const int np = gnn_num_params();
    k_gnn_reduce<<<(np + 31) / 32 + 1, 256, 0, s>>>(a.part, nblk, a.ldp, np, grad, a.lpart, lgrid, loss_dev);
    return cudaGetLastError();
}

cudaError_t gnn_adam(float *theta, const float *grad, float *m, float *v, int cnt, double lr, int step,
                     cudaStream_t s) {
    const double b1 = 0.9, b2 = 0.999;
    const double c1 = 1.0 - std::pow(b1, step), c2 = 1.0 - std::pow(b2, step);
    k_gnn_adam<<<(cnt + 255) / 256, 256, 0, s>>>(theta, grad, m, v, cnt, float(lr), float(b1), float(b2), 1e-8f,
                                                 float(c1), float(c2));
    return cudaGetLastError();
}

#define ALM_GNN_INST(T)                                                                                             \
    template cudaError_t gnn_forward<T>(const GnnGraph &, const GnnParams &, uint64_t, GnnActs<T> &, float *,      \
                                        float *, bool, int, cudaStream_t);                                                \
    template cudaError_t gnn_loss_grad<T>(const GnnGraph &, const GnnParams &, float *, GnnActs<T> &,              \
                                          const float *, const float *, const float *, const double *,             \
                                          const double *, double, double, double, double *, int, cudaStream_t);
ALM_GNN_INST(float)
ALM_GNN_INST(__nv_bfloat16)

}  // namespace alm
