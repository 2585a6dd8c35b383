// Hot-path kernels of the ALM-BM inner loop (arXiv 2505.15775, Eq. AL-BM, Alg. 1):
//
//   k_eval       A(RR^T) and <C, RR^T> (SDDMM v_p = r_i . r_j over the aggregated
//                pattern) with the direct scatter of selector constraints into A(X);
//                for problems whose constraints are all diagonal selectors (MaxCut)
//                also the dual update w = y - sigma(A(X) - b), diag(S) and the L / KKT
//                reductions                                            [hot path (a)]
//   k_gen        A(RR^T)_k of the general (multi-entry) constraints, or their a1, a2
//   k_dual_slack w, the L / KKT reductions and S = C - A^*(w) (general problems)
//   k_spmm       G = 2 S R (+ the low-rank part of C), ||G||^2 and the CG inner
//                products                                              [hot path (b)]
//   k_dir        D = -G + beta D
//   k_ls         the quartic phi(alpha) = L(R + alpha D): a1 = A(RD^T + DR^T),
//                a2 = A(DD^T), <S, RD^T + DR^T>, <S, DD^T> in one pass over R and D,
//                FP64 coefficients and the exact minimiser            [hot path (c)]
//   k_axpy       R += alpha D
//
// Work decomposition.  LANES lanes hold one row of R (lane l the 16-byte vector of columns
// [l W, l W + W), W = 4 floats or 2 doubles), so a gathered row is one coalesced
// 16*LANES-byte read.  SP such subgroups share a row of the pattern (k_spmm, k_ls, k_inner_off):
// subgroup s takes its entries s, s + SP, .., and a row group is LANES x SP lanes.  SP is
// a whole warp's worth when the rows are long, or too few to fill the chip, else one (wide_spmm,
// wide_ls): with one subgroup a row of 80 entries is a serial walk and 10,000 rows at
// rank 3 fill 40 of 152 multiprocessors.  Rows above kHeavyRow entries
// (heavy-tailed graphs) would still be one warp's serial walk: the SpMM's are summed
// beforehand, kHeavySeg entries by a CTA (k_spmm_heavy); the SDDMMs' sums are scalars, so k_ls and
// k_inner_off cut their rows into segments of kUpSeg entries that any row group takes, and k_eval
// takes the entries one by one.
// In FP32, against one subgroup a row and two rows a group: alm_grad on a Kronecker graph of
// 2^16 rows at r = 32 1.62 -> 0.14 ms.
//
// Precision.  FP64 arithmetic is scarce on GB300, so in the FP32 form every per-entry
// product and every per-thread partial sum is FP32; partials are promoted to FP64 once
// per thread, summed per block in FP64 and over blocks in FP64 by the last block to
// finish (a fixed order: results are deterministic).  The dual w and the constraint
// residuals are FP64 throughout.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <mutex>
#include <unordered_map>

#include "sparse_common.cuh"

namespace alm {

// ---------------------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------------------

// The block's share of X^T u_l of the low-rank terms (u_l in FP64) into part[l*kMaxRank + col],
// from a pass of its own over the rows with LANES lanes a row: FP64 instructions cost the same
// for one active lane as for 32, so the split row groups of the kernels would pay SP times.
template <typename T, int LANES>
__device__ __forceinline__ void block_lr_cols(const SparseView<T> &v, const T *__restrict__ X, int r, int ldr,
                                              double *part, double *shm) {
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int gl = lane & (LANES - 1);
    const bool active = gl * W < r;
    for (int l = 0; l < v.lr_k; ++l) {
        double acc[W];
#pragma unroll
        for (int k = 0; k < W; ++k) acc[k] = 0.0;
        for (int64_t i = int64_t(blockIdx.x) * (kBlock / LANES) + threadIdx.x / LANES; i < v.n;
             i += int64_t(gridDim.x) * (kBlock / LANES)) {
            const V x = mask_tail(load_row(X, i, ldr, gl, active), gl * W, r);
            const double u = v.lr_u[int64_t(l) * v.n + i];
#pragma unroll
            for (int k = 0; k < W; ++k) acc[k] = fma(u, double(comp(x, k)), acc[k]);
        }
#pragma unroll
        for (int k = 0; k < W; ++k)
#pragma unroll
            for (int o = 16; o >= LANES; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
        __syncthreads();
        if (lane < LANES)
#pragma unroll
            for (int k = 0; k < W; ++k)
                if (lane * W + k < kMaxRank) shm[warp * 32 + lane * W + k] = acc[k];
        __syncthreads();
        if (threadIdx.x < kMaxRank) {
            double t = 0.0;
            if (threadIdx.x < LANES * W)
                for (int q = 0; q < nw; ++q) t += shm[q * 32 + threadIdx.x];
            part[l * kMaxRank + threadIdx.x] = t;
        }
    }
}

// In the last block: z[l][col] = sum over the blocks of part (one warp per column, lanes over
// the blocks in a fixed order), zero from column r on; visible to the block on return
__device__ __forceinline__ void sum_lr_cols(const double *part, int nl, int r, double (*z)[kMaxRank]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int t = warp; t < nl * kMaxRank; t += nw) {
        const int col = t % kMaxRank;
        double a = 0.0;
        if (col < r)
            for (int b = lane; b < int(gridDim.x); b += 32) a += __ldcg(part + size_t(b) * kPartStride + t);
        a = warp_sum(a);
        if (lane == 0) z[t / kMaxRank][col] = a;
    }
    __syncthreads();
}

template <typename T, int LANES>
__device__ __forceinline__ void slack_row(const SparseView<T> &v, int64_t i, T xh, T xl, T sigma) {
    const int k = v.d_sel_k[i];
    T dh = v.base_hi[i], dl = v.base_lo ? v.base_lo[i] : T(0);
    if (k >= 0) {
        const T a = sizeof(T) == 8 ? T(v.d_sel_a[i]) : T(v.d_sel_af[i]);
        // a x = (ph + pe) + a xl exactly up to the last term's rounding
        const T ph = a * xh;
        const T pe = fma(a, xh, -ph) + a * xl;
        // res = (ph - b_hi) + (pe - b_lo), the first difference with two-sum
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
    v.d_s[i] = dh;
    if (v.d_s_lo) v.d_s_lo[i] = dl;
    if (v.ls_rec) v.ls_rec[i].ds = dh;
}

// STEP: first apply the pending step R += alpha D of the previous line search (alpha = 0
// at the start of an inner solve), so that no separate update pass is needed.
// Four rows per group and iteration are loaded before any of them is used.
template <typename T, int LANES, bool STEP>
__global__ void __launch_bounds__(kBlock, 4) k_inner_slack(SparseView<T> v, T *__restrict__ R, const T *__restrict__ D,
                                                        int r, int ldr, const DevState *st, const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    constexpr int B = 4;
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LANES - 1);
    const unsigned gmask = group_mask<LANES>(lane);
    const int gpb = kBlock / LANES;
    const int64_t ng = int64_t(gridDim.x) * gpb;
    const bool active = gl * W < r;
    const bool writer = gl * W < ldr;
    const T sigma = T(st->sigma);
    const T alpha = STEP ? T(st->alpha) : T(0);
    const bool step = STEP && alpha != T(0);
    for (int64_t i0 = int64_t(blockIdx.x) * gpb + threadIdx.x / LANES; i0 < v.n; i0 += B * ng) {
        V rv[B];
        int64_t row[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            row[b] = i0 + b * ng;
            const bool ok = row[b] < v.n;
            rv[b] = ok && writer ? ld(R + row[b] * ldr + gl * W) : vzero(T());
        }
        if (step) {
            V dv[B];
#pragma unroll
            for (int b = 0; b < B; ++b) dv[b] = row[b] < v.n && writer ? ld(D + row[b] * ldr + gl * W) : vzero(T());
#pragma unroll
            for (int b = 0; b < B; ++b) {
                rv[b] = fma4(alpha, dv[b], rv[b]);
                if (row[b] < v.n && writer) stv(R + row[b] * ldr + gl * W, rv[b]);
            }
        }
#pragma unroll
        for (int b = 0; b < B; ++b) {
            if (row[b] >= v.n) break;  // group-uniform
            T xh, xl;
            norm2_pair(mask_tail(rv[b], gl * W, r), gmask, LANES, xh, xl);
            if (gl == 0) slack_row<T, LANES>(v, row[b], xh, xl, sigma);
        }
    }
}

// FP64 form of k_inner_slack.  FP64 instructions bound it (a warp's takes 64 cycles, and a row's
// scalar work cost as many on a leader lane as the row's 32 elements): a warp takes LANES rows
// per row group, its lanes' partial squares are reduced for all of them at once (LANES - 1
// additions instead of LANES log2 LANES), which leaves lane t with row t's sum, and every lane
// then does one row's scalars, the two divisions of the preconditioner among them (k_spmm_ell
// reads them back).  201,601 rows, r = 32: 188 -> 60 us.
template <int LANES, bool STEP>
__global__ void __launch_bounds__(kBlock) k_inner_slack64(SparseView<double> v, double *__restrict__ R,
                                                          const double *__restrict__ D, int r, int ldr,
                                                          const DevState *st, const int *done) {
    if (*done) return;
    constexpr int RW = 32 / LANES;
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LANES - 1);
    const bool writer = gl * 2 < ldr;
    const double sigma = st->sigma;
    const double alpha = STEP ? st->alpha : 0.0;
    const bool step = STEP && alpha != 0.0;
    const int64_t nw = int64_t(gridDim.x) * (kBlock / 32);
    for (int64_t t0 = (int64_t(blockIdx.x) * (kBlock / 32) + (threadIdx.x >> 5)) * 32; t0 < v.n; t0 += nw * 32) {
        double p[LANES];
#pragma unroll
        for (int t = 0; t < LANES; ++t) {
            const int64_t i = t0 + t * RW + lane / LANES;
            double2 x = make_double2(0.0, 0.0);
            if (writer && i < v.n) {
                x = ld(R + i * ldr + gl * 2);
                if (step) {
                    x = fma4(alpha, ld(D + i * ldr + gl * 2), x);
                    stv(R + i * ldr + gl * 2, x);
                }
            }
            x = mask_tail(x, gl * 2, r);
            p[t] = fma(x.x, x.x, x.y * x.y);
        }
#pragma unroll
        for (int s = LANES / 2; s > 0; s >>= 1) {
            const bool up = gl & s;
#pragma unroll
            for (int u = 0; u < s; ++u) {
                const double give = up ? p[u] : p[u + s], keep = up ? p[u + s] : p[u];
                p[u] = keep + __shfl_xor_sync(0xffffffffu, give, s);
            }
        }
        const int64_t i = t0 + gl * RW + lane / LANES;
        if (i < v.n) {
            slack_row<double, LANES>(v, i, p[0], 0.0, sigma);
            if (v.pc_rec && st->precond) {
                double sdi = v.d_s[i];
                sdi = sdi > st->pc_floor ? sdi : st->pc_floor;
                const double a = v.d_sel_k[i] >= 0 ? v.d_sel_a[i] : 0.0;
                const double ka = 4.0 * sigma * a * a;
                v.pc_rec[i] = make_double2(1.0 / (2.0 * sdi), ka / (2.0 * sdi + ka * p[0]));
            }
        }
    }
}

// base_i = C_ii - a_i y_k(i) (rows without a diagonal selector: C_ii), as a float pair
template <typename T>
__global__ void __launch_bounds__(kBlock) k_prep_base(SparseView<T> v, const double *__restrict__ y,
                                                      T *__restrict__ base_hi, T *__restrict__ base_lo) {
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < v.n; i += int64_t(gridDim.x) * blockDim.x) {
        double d = double(v.d_c[i]);
        const int k = v.d_sel_k[i];
        if (k >= 0) d -= v.d_sel_a[i] * y[k];
        T hi, lo;
        split_pair(d, hi, lo);
        base_hi[i] = hi;
        if (base_lo) base_lo[i] = lo;
        if (v.step_rec) {
            v.step_rec[i].base_hi = float(hi);
            v.step_rec[i].base_lo = float(lo);
        }
    }
}

// ---------------------------------------------------------------------------------------
// (a) constraint map + <C, RR^T> (+ fused dual update for diagonal-selector problems)
// ---------------------------------------------------------------------------------------
// The rows' FP64 work goes through a warp at a time; the strict upper entries are taken two per
// row group and round from the whole pattern, whatever rows they lie in: four independent gathers
// a lane, and no row sets the time.  Walking the entries by rows instead (subgroups of a warp sharing
// the long ones) was slower nearly everywhere: ER(60,000) of degree 40, r = 32, FP32 151 us a call
// against 102; a Kronecker graph of 2^13 rows, r = 1 110 against 64; matrix completion, n = 1e4, r = 3,
// FP64 123 against 101.  BYROW is what is left of it: FP32 factors that do not stay in L2 and rows of at
// most two upper entries, where it reads R twice instead of 2.5 times (eval_by_row has the line).
template <typename T, int LANES, bool BYROW, bool OFFSEL, bool LR, bool FUSED>
__global__ void __launch_bounds__(kBlock) k_eval(SparseView<T> v, const T *__restrict__ R, int r, int ldr,
                                                 double *__restrict__ AX, const double *__restrict__ y,
                                                 double *__restrict__ w, int nb, double sigma_arg, HostResult *res,
                                                 DevState *st, double *partials, const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    constexpr int U = 2;  // entries per row group and round
    __shared__ double shm[32 * 32];
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LANES - 1);
    const unsigned gmask = group_mask<LANES>(lane);
    const int64_t g0 = int64_t(blockIdx.x) * (kBlock / LANES) + threadIdx.x / LANES;
    const int64_t ng = int64_t(gridDim.x) * (kBlock / LANES);
    const bool active = gl * W < r;
    const double sigma = FUSED ? (sigma_arg >= 0.0 ? sigma_arg : st->sigma) : 0.0;
    T pc = T(0);
    double pyres = 0.0, pres2 = 0.0, pbw = 0.0;

    // BYROW: strict upper entries e0 .. e1-1 of a row (ri its masked vector)
    auto upper = [&](V ri, int64_t i, int e0, int e1) {
        T acc = T(0);
        for (int e = e0; e < e1; e += U) {
            int j[U];
            T c[U];
            V x[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const bool in = e + k < e1;
                j[k] = in ? v.up_col[e + k] : int(i);
                c[k] = in ? v.up_c[e + k] : T(0);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) x[k] = load_row(R, j[k], ldr, gl, active);
#pragma unroll
            for (int k = 0; k < U; ++k) acc += c[k] * dot(ri, x[k]);
        }
        pc += T(2) * acc;
    };
    // A warp takes nb rows per row group and keeps row t's |r_i|^2 in the group's lane t; then
    // every lane does one row's FP64 work.  An FP64 instruction holds a warp 64 cycles whatever
    // the number of active lanes, and a row takes about 16: one leader lane per row at a time
    // cost 206 us on 1e6 rows at r = 32, of which the memory traffic is 60.
    constexpr int RW = 32 / LANES;  // row groups of a warp
    const int x = gl;
    const int64_t tile = int64_t(RW) * nb;
    const int64_t nw = int64_t(gridDim.x) * (kBlock / 32);
    for (int64_t t0 = (int64_t(blockIdx.x) * (kBlock / 32) + (threadIdx.x >> 5)) * tile; t0 < v.n; t0 += nw * tile) {
        T kh = T(0), kl = T(0);
        for (int t = 0; t < nb; ++t) {
            const int64_t i = t0 + int64_t(t) * RW + lane / LANES;
            const bool in = i < v.n;  // group-uniform
            const V ri = mask_tail(load_row(R, in ? i : 0, ldr, gl, active && in), gl * W, r);
            T hi, lo;
            norm2_pair(ri, gmask, LANES, hi, lo);  // compensated in FP32
            if (x == t) {
                kh = hi;
                kl = lo;
            }
            if (BYROW && in && !v.diag_only) {
                const int e0 = v.up_ptr[i];
                upper(ri, i, e0, min(v.up_ptr[i + 1], e0 + kUpSeg));
            }
        }
        __syncwarp();
        const int64_t i = t0 + int64_t(x) * RW + lane / LANES;
        if (x < nb && i < v.n) {
            const double viid = double(kh) + double(kl);
            const T cii = v.d_c[i];
            pc += cii * T(viid);
            const int k = v.d_sel_k[i];
            if (k >= 0) {
                const double a = v.d_sel_a[i];
                const double ax = a * viid;
                AX[k] = ax;
                if (FUSED) {
                    const double res = ax - v.b[k];
                    const double wk = y[k] - sigma * res;
                    w[k] = wk;
                    store_slack_diag(v, i, double(cii) - wk * a);
                    pyres += y[k] * res;
                    pres2 += res * res;
                    pbw += v.b[k] * wk;
                }
            } else if (FUSED) {
                store_slack_diag(v, i, double(cii));
            }
        }
        __syncwarp();
    }
    if (BYROW) {
        for (int64_t q = g0; q < v.n_useg && !v.diag_only; q += ng) {  // the rest of the long rows
            const int i = v.us_row[q], e0 = v.us_e0[q], e1 = min(v.up_ptr[i + 1], e0 + kUpSeg);
            upper(mask_tail(load_row(R, i, ldr, gl, active), gl * W, r), i, e0, e1);
        }
    } else if (!v.diag_only) {
        for (int64_t e = g0; e < v.nnz_u; e += U * ng) {
            V a[U], b[U];
            T c[U];
            bool has[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                has[k] = e + k * ng < v.nnz_u;  // group-uniform
                const int64_t q = has[k] ? e + k * ng : e;
                const int i = v.up_row[q], j = v.up_col[q];
                c[k] = has[k] ? v.up_c[q] : T(0);
                a[k] = load_row(R, i, ldr, gl, active);
                b[k] = load_row(R, j, ldr, gl, active);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                a[k] = mask_tail(a[k], gl * W, r);
                if (OFFSEL) {
                    T hi, lo;
                    dot_pair(a[k], b[k], hi, lo);
                    if (sizeof(T) == 4) pc += T(2) * c[k] * hi;  // FP64: the leader's whole sum, one FMA
                    pair_group_sum<LANES>(hi, lo, gmask);
                    if (gl == 0 && has[k]) {
                        const int64_t q = e + k * ng;
                        const int s = v.up_sel_k[q];
                        if (sizeof(T) == 8) {
                            pc = fma(T(2) * c[k], hi, pc);
                            if (s >= 0) AX[s] = double(v.up_sel_a2[q]) * double(hi);
                        } else if (s >= 0) {
                            AX[s] = 2.0 * v.up_sel_a[q] * (double(hi) + double(lo));
                        }
                    }
                } else {
                    pc += T(2) * c[k] * dot(a[k], b[k]);
                }
            }
        }
    }
    double *part = partials + size_t(blockIdx.x) * kPartStride;
    if (FUSED) {
        const double vals[4] = {double(pc), pyres, pres2, pbw};
        block_partials<4>(vals, part, shm);
    } else {
        const double vals[1] = {double(pc)};
        block_partials<1>(vals, part, shm);
    }
    if (LR) block_lr_cols<T, LANES>(v, R, r, ldr, part + 4, shm);
    if (!last_block(&st->counter[CNT_EVAL])) return;
    double tot[4] = {0.0, 0.0, 0.0, 0.0};
    if (FUSED) {
        sum_partials_n<4>(partials, tot, shm);
    } else {
        double t1[1];
        sum_partials_n<1>(partials, t1, shm);
        tot[0] = t1[0];
    }
    if (LR) sum_lr_cols(partials + 4, v.lr_k, r, st->z);
    if (threadIdx.x == 0) {
        double c = tot[0];
        for (int l = 0; LR && l < v.lr_k; ++l) {
            double zz = 0.0;
            for (int col = 0; col < r; ++col) zz += st->z[l][col] * st->z[l][col];
            c += v.lr_s[l] * zz;
        }
        st->c0 = c;
        if (FUSED) {
            st->yres = tot[1];
            st->res2 = tot[2];
            st->bw = tot[3];
            const double L = c - tot[1] + 0.5 * sigma * tot[2];
            st->L = L;
            if (sigma_arg >= 0.0) {  // a primitive: the state that k_set_state prepares for a solve
                st->sigma = sigma;
                st->status = isfinite(L) ? 0 : ALM_ERR_NUMERIC;
                if (res) {
                    res->L = L;
                    res->c0 = c;
                    res->status = st->status;
                    __threadfence_system();
                }
            } else if (!isfinite(L)) {
                st->status = ALM_ERR_NUMERIC;
                st->done = 1;
            }
        }
    }
}

// ---------------------------------------------------------------------------------------
// General (multi-entry) constraints: A(X)_k = sum over its entries of kappa a (r_i . r_j)
// (LS: a1_k = A(RD^T + DR^T)_k and a2_k = A(DD^T)_k into g_a1, g_a2).  The entries are cut
// into chunks of kGenChunk, one CTA each, so that a constraint on every row (the trace of a
// theta SDP) fills the chip instead of one CTA; a row group of LANES lanes reads each row as
// one coalesced vector per lane and keeps its columns' share of the sum in FP64 (no reduction
// per entry).  The last chunk of a constraint to finish adds up the chunks in order.
// With one CTA per constraint and a thread per entry walking its columns the trace over 20,000
// rows at r = 29 took 575 us, its line-search form 1189 us; alm_linesearch on that theta SDP
// went from 2.03 to 0.30 ms with the chunks.
// ---------------------------------------------------------------------------------------
template <typename T, int LANES, bool LS>
__global__ void __launch_bounds__(kBlock) k_gen(SparseView<T> v, const T *__restrict__ R, const T *__restrict__ D,
                                                int r, int ldr, double *__restrict__ AX, const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    __shared__ double shm[64];
    __shared__ bool last;
    const int gl = threadIdx.x & (LANES - 1);
    const bool active = gl * W < r;
    for (int c = blockIdx.x; c < v.n_gchunk; c += gridDim.x) {
        const int g = v.gc_con[c], c0 = v.g_cptr[g], nc = v.g_cptr[g + 1] - c0;
        const int e0 = v.g_ptr[g] + (c - c0) * kGenChunk;
        const int len = min(v.g_ptr[g + 1] - e0, kGenChunk);
        double a1 = 0.0, a2 = 0.0;
        for (int q = threadIdx.x / LANES; q < len; q += kBlock / LANES) {  // by offset: e0 + q may be near 2^31
            const int t = e0 + q, i = v.g_i[t], j = v.g_j[t];
            const double ka = (i == j ? 1.0 : 2.0) * v.g_a[t];
            const V ri = mask_tail(load_row(R, i, ldr, gl, active), gl * W, r);
            const V rj = load_row(R, j, ldr, gl, active);
            if (LS) {
                const V di = mask_tail(load_row(D, i, ldr, gl, active), gl * W, r);
                const V dj = load_row(D, j, ldr, gl, active);
                a1 = fma(ka, double(dot(ri, dj) + dot(di, rj)), a1);
                a2 = fma(ka, double(dot(di, dj)), a2);
            } else {
                T hi, lo;
                dot_pair(ri, rj, hi, lo);
                a1 = fma(ka, double(hi), a1);
                if (sizeof(T) == 4) a1 = fma(ka, double(lo), a1);
            }
        }
        a1 = block_sum(a1, shm);
        if (LS) a2 = block_sum(a2, shm);
        if (nc > 1) {
            if (threadIdx.x == 0) {
                v.g_part[2 * c] = a1;
                v.g_part[2 * c + 1] = a2;
                __threadfence();
                last = atomicAdd(v.g_cnt + g, 1u) == unsigned(nc - 1);
                if (last) v.g_cnt[g] = 0u;
            }
            __syncthreads();
            if (!last) continue;  // block-uniform
            __threadfence();
            double s1 = 0.0, s2 = 0.0;
            for (int q = threadIdx.x; q < nc; q += kBlock) {
                s1 += __ldcg(v.g_part + 2 * (c0 + q));
                if (LS) s2 += __ldcg(v.g_part + 2 * (c0 + q) + 1);
            }
            a1 = block_sum(s1, shm);
            if (LS) a2 = block_sum(s2, shm);
        }
        if (threadIdx.x == 0) {
            if (LS) {
                v.g_a1[g] = a1;
                v.g_a2[g] = a2;
            } else {
                AX[v.g_con[g]] = a1;
            }
        }
        __syncthreads();  // `last` is reused
    }
}

// ---------------------------------------------------------------------------------------
// dual update, L and KKT reductions, slack values S = C - A^*(w) (general problems)
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kBlock) k_dual_slack(SparseView<T> v, const double *__restrict__ y,
                                                       const double *__restrict__ AX, double *__restrict__ w,
                                                       const int2 *__restrict__ up_slot, DevState *st,
                                                       double *partials, const int *done) {
    if (*done) return;
    __shared__ double shm[64];
    const double sigma = st->sigma;
    const int64_t tid = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t nt = int64_t(gridDim.x) * blockDim.x;
    double pyres = 0.0, pres2 = 0.0, pbw = 0.0;
    for (int64_t k = tid; k < v.m; k += nt) {
        const double res = AX[k] - v.b[k];
        const double wk = y[k] - sigma * res;
        w[k] = wk;
        pyres += y[k] * res;
        pres2 += res * res;
        pbw += v.b[k] * wk;
    }
    // w_k is recomputed where another block owns k
#define WOF(k) (y[(k)] - sigma * (AX[(k)] - v.b[(k)]))
    for (int64_t i = tid; i < v.n; i += nt) {
        double s = double(v.d_c[i]);
        const int k = v.d_sel_k[i];
        if (k >= 0) s -= WOF(k) * v.d_sel_a[i];
        if (v.gd_ptr)
            for (int t = v.gd_ptr[i]; t < v.gd_ptr[i + 1]; ++t) s -= WOF(v.gd_k[t]) * v.gd_a[t];
        store_slack_diag(v, i, s);
    }
    if (v.off_dynamic) {
        for (int64_t e = tid; e < v.nnz_u; e += nt) {
            double s = double(v.up_c[e]);
            if (v.has_off_sel) {
                const int k = v.up_sel_k[e];
                if (k >= 0) s -= WOF(k) * v.up_sel_a[e];
            }
            if (v.gu_ptr)
                for (int t = v.gu_ptr[e]; t < v.gu_ptr[e + 1]; ++t) s -= WOF(v.gu_k[t]) * v.gu_a[t];
            const T sv = T(s);
            v.up_s[e] = sv;
            const int2 sl = up_slot[e];
            v.f_val[sl.x] = sv;
            v.f_val[sl.y] = sv;
        }
    }
#undef WOF
    const double vals[3] = {pyres, pres2, pbw};
    block_partials<3>(vals, partials + size_t(blockIdx.x) * kPartStride, shm);
    if (!last_block(&st->counter[CNT_DUAL])) return;
    const double yres = sum_partials(partials, 0, shm);
    const double res2 = sum_partials(partials, 1, shm);
    const double bw = sum_partials(partials, 2, shm);
    if (threadIdx.x == 0) {
        st->yres = yres;
        st->res2 = res2;
        st->bw = bw;
        st->L = st->c0 - yres + 0.5 * sigma * res2;
        if (!isfinite(st->L)) {
            st->status = ALM_ERR_NUMERIC;
            st->done = 1;
        }
    }
}

// Per outer iteration: C_ij - a y_k of every strict upper entry as a pair
template <typename T>
__global__ void __launch_bounds__(kBlock) k_prep_off(SparseView<T> v, const double *__restrict__ y) {
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < v.nnz_u; e += int64_t(gridDim.x) * blockDim.x) {
        double d = double(v.up_c[e]);
        const int k = v.up_sel_k[e];
        if (k >= 0) d -= v.up_sel_a[e] * y[k];
        T hi, lo;
        split_pair(d, hi, lo);
        v.ob_hi[e] = hi;
        v.ob_lo[e] = lo;
    }
}

// (h + l) + sigma m (c x - b) as a normalised pair; x, b and sigma are pairs, m and c floats.  Every
// product and sum keeps its rounding error, so that the result has its own relative accuracy also
// where the two terms cancel (a multiplier close to sigma times a large residual).
__device__ __forceinline__ void selector_slack(float h, float l, float m, float c, float xh, float xl, float bh,
                                               float bl, float sh, float sl, float &oh, float &ol) {
    const float ph = c * xh;
    const float pe = fmaf(c, xh, -ph) + c * xl;
    const float s0 = ph - bh;
    const float bb = s0 - ph;
    const float r0 = ((ph - (s0 - bb)) + (-bh - bb)) + (pe - bl);
    const float kh = sh * m;
    const float kl = fmaf(sh, m, -kh) + sl * m;
    const float ch = kh * s0;
    const float cl = fmaf(kh, s0, -ch) + fmaf(kh, r0, kl * s0);
    const float s1 = h + ch;
    const float b1 = s1 - h;
    const float e1 = l + (cl + ((h - (s1 - b1)) + (ch - b1)));
    oh = s1 + e1;
    ol = e1 - (oh - s1);
}
__device__ __forceinline__ void selector_slack(double h, double, double m, double c, double x, double, double b, double,
                                               double sigma, double, double &oh, double &ol) {
    oh = fma(sigma * m, fma(c, x, -b), h);
    ol = 0.0;
}

// Slack update of the inner loop when every constraint is a selector and some are off the
// diagonal (matrix completion): S_ij = (C_ij - a y_k) + sigma a (2 a r_i.r_j - b_k) in float
// pairs (selector_slack), in one pass over the upper pattern.  k_eval and
// k_dual_slack (still what ends an inner solve) put the values through FP64 A(X) and w, some 15
// FP64 instructions an entry at 64 cycles a warp: together 85 us on 829,000 entries
// at rank 3 (cold caches), this 21 us (18 with sigma and the products rounded to floats, which loses S
// where its terms cancel); 32 inner steps there 4.49 -> 3.00 ms with it.
template <typename T, int LANES, int SP>
__global__ void __launch_bounds__(kBlock) k_inner_off(SparseView<T> v, const T *__restrict__ R, int r, int ldr,
                                                      const DevState *st, const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    constexpr int GW = LANES * SP;
    constexpr int U = 2;
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LANES - 1), sub = (lane & (GW - 1)) / LANES;
    const unsigned gmask = group_mask<GW>(lane);
    const int64_t g0 = int64_t(blockIdx.x) * (kBlock / GW) + threadIdx.x / GW;
    const int64_t ng = int64_t(gridDim.x) * (kBlock / GW);
    const bool active = gl * W < r;
    T sh, sl;
    split_pair(st->sigma, sh, sl);
    auto upper = [&](V ri, int64_t i, int e0, int e1) {
        for (int e = e0 + sub; e < e1 + sub; e += U * SP) {  // group-uniform trip count
            int j[U];
            V x[U];
#pragma unroll
            for (int k = 0; k < U; ++k) j[k] = e + k * SP < e1 ? v.up_col[e + k * SP] : int(i);
#pragma unroll
            for (int k = 0; k < U; ++k) x[k] = load_row(R, j[k], ldr, gl, active);
#pragma unroll
            for (int k = 0; k < U; ++k) {
                T xh, xl;
                dot_pair(ri, x[k], xh, xl);
                pair_group_sum<LANES>(xh, xl, gmask);
                const int q = e + k * SP;
                if (gl == 0 && q < e1) {
                    const T a = v.up_sel_t[q];  // 0 without a selector
                    T s, lo;
                    selector_slack(v.ob_hi[q], v.ob_lo[q], a, a + a, xh, xl, v.obb_hi[q], v.obb_lo[q], sh, sl, s, lo);
                    v.up_s[q] = s;
                    const int2 at = v.up_slot[q];
                    v.f_val[at.x] = s;
                    v.f_val[at.y] = s;
                }
            }
        }
    };
    for (int64_t i = g0; i < v.n; i += ng) {
        const V ri = mask_tail(load_row(R, i, ldr, gl, active), gl * W, r);
        const int e0 = v.up_ptr[i], e1 = min(v.up_ptr[i + 1], e0 + kUpSeg);
        T xh, xl;
        norm2_pair(ri, gmask, LANES, xh, xl);
        if (gl == 0 && sub == 0) {
            T dh = v.base_hi[i], dl = v.base_lo ? v.base_lo[i] : T(0);
            if (v.d_sel_k[i] >= 0) {
                const T a = sizeof(T) == 8 ? T(v.d_sel_a[i]) : T(v.d_sel_af[i]);
                selector_slack(dh, dl, a, a, xh, xl, v.b_hi[i], v.b_lo ? v.b_lo[i] : T(0), sh, sl, dh, dl);
            }
            v.d_s[i] = dh;
            if (v.d_s_lo) v.d_s_lo[i] = dl;
        }
        upper(ri, i, e0, e1);
    }
    for (int64_t q = g0; q < v.n_useg; q += ng) {
        const int i = v.us_row[q], e0 = v.us_e0[q], e1 = min(v.up_ptr[i + 1], e0 + kUpSeg);
        upper(mask_tail(load_row(R, i, ldr, gl, active), gl * W, r), i, e0, e1);
    }
}

// ---------------------------------------------------------------------------------------
// (b) G = 2 S R
//   MODE 0: gradient only (and ||G||^2)
//   MODE 1: inner CG step: also <G, G_old> (G is updated in place) and <G, D_old>, the
//           stop test ||G|| <= tau and the Polak-Ribiere+ coefficient
// ---------------------------------------------------------------------------------------
// Off-diagonal sums of the rows above kHeavyRow entries, segments of kHeavySeg of them by one CTA
// each, into hs_sum (the accumulator's state per column vector; k_spmm adds a row's up).  With one
// CTA per row the longest row set the time (129 us at 8.6% of the SM rate): alm_grad on a Kronecker
// graph of 2^16 rows at r = 32, FP32, 268 -> 170 us.
template <typename T, int LANES>
__global__ void __launch_bounds__(kBlock) k_spmm_heavy(SparseView<T> v, const T *__restrict__ R, int r, int ldr,
                                                       const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    using Acc = typename AccOf<T>::type;
    constexpr int W = VecT<T>::W;
    constexpr int U = 4;
    constexpr int NSUB = kBlock / LANES;
    __shared__ __align__(16) T sh[kBlock / 32][LANES][Acc::kWords * W];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gl = lane & (LANES - 1);
    const bool active = gl * W < r;
    for (int q = blockIdx.x; q < v.n_hseg; q += gridDim.x) {
        const int i = v.hs_row[q], e0 = v.hs_e0[q];
        const int len = min(v.f_ptr[i + 1] - e0, kHeavySeg);
        Acc acc;
        acc.init();
        for (int t = threadIdx.x / LANES; t < len; t += U * NSUB) {  // by offset: e0 + t may be near 2^31
            int j[U];
            T c[U];
            V x[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const bool in = t + k * NSUB < len;
                j[k] = in ? v.f_col[e0 + t + k * NSUB] : i;
                c[k] = in ? v.f_val[e0 + t + k * NSUB] : T(0);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) x[k] = load_row(R, j[k], ldr, gl, active);
#pragma unroll
            for (int k = 0; k < U; ++k) acc.add(c[k], x[k]);
        }
        __syncwarp();
        acc.template merge<LANES, 32>(0xffffffffu);
        if (lane < LANES) acc.store(sh[warp][lane]);
        __syncthreads();
        if (threadIdx.x < LANES) {
            for (int ww = 1; ww < kBlock / 32; ++ww) acc.add_stored(sh[ww][lane]);
            acc.store(v.hs_sum + (int64_t(q) * LANES + lane) * (Acc::kWords * W));
        }
        __syncthreads();
    }
}

template <typename T, int LANES, int SP, bool LR, int MODE>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 8 ? 3 : 4) k_spmm(SparseView<T> v, const T *__restrict__ R,
                                                                      int r, int ldr, T *G, const T *D, HostResult *res,
                                                                      DevState *st, double *partials, const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    using Acc = typename AccOf<T>::type;
    constexpr int W = VecT<T>::W;
    constexpr int GW = LANES * SP;
    constexpr int U = 4;  // entries per subgroup and round
    __shared__ double shm[64];
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LANES - 1), sub = (lane & (GW - 1)) / LANES;
    const unsigned gmask = group_mask<GW>(lane);
    const int64_t g0 = int64_t(blockIdx.x) * (kBlock / GW) + threadIdx.x / GW;
    const int64_t ng = int64_t(gridDim.x) * (kBlock / GW);
    const bool active = gl * W < r;
    const bool writer = sub == 0 && gl * W < ldr;
    V zl[LR ? kMaxLR : 1];
    if (LR)
        for (int l = 0; l < v.lr_k; ++l) {
            T zz[W];
            for (int k = 0; k < W; ++k) {
                const int col = gl * W + k;
                zz[k] = (col < r) ? T(v.lr_s[l] * st->z[l][col]) : T(0);
            }
            if constexpr (W == 4) zl[l] = make_float4(zz[0], zz[1], zz[2], zz[3]);
            else zl[l] = make_double2(zz[0], zz[1]);
        }
    T pgg = T(0), pgg_lo = T(0), pgo = T(0), pgd = T(0), pzg = T(0);
    const bool pc = MODE == 1 && st->precond;
    const T sig = T(st->sigma);
    const T pc_floor = T(st->pc_floor);
    for (int64_t i = g0; i < v.n; i += ng) {
        const V ri = mask_tail(load_row(R, i, ldr, gl, active), gl * W, r);
        const int e0 = v.f_ptr[i], len = v.f_ptr[i + 1] - e0;
        const T ds = v.d_s[i], dlo = v.d_s_lo ? v.d_s_lo[i] : T(0);
        V gold = vzero(T()), dold = vzero(T());
        if (MODE == 1 && active && sub == 0) {
            gold = ld(G + i * ldr + gl * W);
            dold = ld(D + i * ldr + gl * W);
        }
        Acc acc;
        acc.init();
        if (sub == 0) {
            acc.add(ds, ri);
            acc.add_lo(dlo, ri);
            if (LR)
                for (int l = 0; l < v.lr_k; ++l) acc.add(T(v.lr_u[int64_t(l) * v.n + i]), zl[l]);
        }
        if (v.n_heavy > 0 && len > kHeavyRow) {  // its entries are summed already
            int a = 0, b = v.n_heavy - 1;
            while (a < b) {
                const int mid = (a + b) / 2;
                if (v.hv_row[mid] < int(i)) a = mid + 1;
                else b = mid;
            }
            const int q1 = v.hv_ptr[a + 1];
#pragma unroll 4
            for (int q = v.hv_ptr[a] + sub; q < q1; q += SP)
                acc.add_stored(v.hs_sum + (int64_t(q) * LANES + gl) * (Acc::kWords * W));
        } else {
            for (int t = sub; t < len; t += U * SP) {  // by offset: e0 + t may be near 2^31
                int j[U];
                T c[U];
                V x[U];
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const bool in = t + k * SP < len;
                    j[k] = in ? v.f_col[e0 + t + k * SP] : int(i);
                    c[k] = in ? v.f_val[e0 + t + k * SP] : T(0);
                }
#pragma unroll
                for (int k = 0; k < U; ++k) x[k] = load_row(R, j[k], ldr, gl, active);
#pragma unroll
                for (int k = 0; k < U; ++k) acc.add(c[k], x[k]);
            }
        }
        __syncwarp(gmask);
        acc.template merge<LANES, GW>(gmask);
        const V g = mask_tail(scale4(T(2), acc.value()), gl * W, r);
        if constexpr (MODE == 0 && sizeof(T) == 4) {  // a few long rows can hold most of |G|^2: a float pair
            if (sub == 0) {
                T h, l;
                dot_pair(g, g, h, l);
                two_sum_acc(pgg, pgg_lo, h);
                pgg_lo += l;
            }
        } else if (sub == 0) {
            pgg += dot(g, g);
        }
        if (MODE == 1) {
            // Row-block Jacobi preconditioner Z = P^{-1} G with P_i = 2 s_i I + 4 sigma a_i^2 r_i r_i^T
            // (the block of the Hessian of L in row i: the S_ii part and the penalty of the
            // diagonal selector a_i e_i e_i^T), inverted by Sherman-Morrison; s_i = S_ii floored.
            V z = g;
            if (pc) {
                const T rg = group_sum<LANES>(dot(ri, g), gmask), rr = group_sum<LANES>(dot(ri, ri), gmask);
                T sdi = ds + dlo;
                sdi = sdi > pc_floor ? sdi : pc_floor;
                const int k = v.d_sel_k[i];
                const T a = k >= 0 ? T(v.d_sel_a[i]) : T(0);
                const T ka = T(4) * sig * a * a;
                const T coef = ka * rg / (T(2) * sdi + ka * rr);
                z = scale4(T(1) / (T(2) * sdi), fma4(-coef, ri, g));
            }
            if (sub == 0) {
                pzg += dot(z, g);
                pgo += dot(g, gold);
                pgd += dot(g, dold);
            }
            if (writer) stv(G + i * ldr + gl * W, z);
        } else if (writer) {
            stv(G + i * ldr + gl * W, g);
        }
    }
    double *part = partials + size_t(blockIdx.x) * kPartStride;
    const double vals[4] = {double(pgg) + double(pgg_lo), double(pgo), double(pgd), double(pzg)};
    block_partials<4>(vals, part, shm);
    if (!last_block(&st->counter[CNT_SPMM])) return;
    double tot[4];
    sum_partials_n<4>(partials, tot, shm);
    if (threadIdx.x == 0) {
        if (MODE == 1) {
            spmm_finish(st, tot[0], tot[1], tot[2], tot[3]);
        } else {
            st->gg = tot[0];
            if (res) {
                res->gg = tot[0];
                __threadfence_system();
            }
        }
    }
}


template <typename T, int LANES, int KF, int MODE>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 8 ? 3 : 4) k_spmm_ell(SparseView<T> v, const T *__restrict__ R, int r, int ldr,
                                                     T *G, const T *D, HostResult *res, DevState *st,
                                                     double *partials, const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    __shared__ double shm[64];
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LANES - 1);
    const unsigned gmask = group_mask<LANES>(lane);
    const int gpb = kBlock / LANES;
    const int64_t ng = int64_t(gridDim.x) * gpb;
    const bool active = gl * W < r;
    const bool writer = gl * W < ldr;
    const bool pc = MODE == 1 && st->precond;
    const T sig = T(st->sigma);
    const T pc_floor = T(st->pc_floor);
    T pgg = T(0), pgo = T(0), pgd = T(0), pzg = T(0);
    int jc[KF];
    T sc[KF];
    int64_t i = int64_t(blockIdx.x) * gpb + threadIdx.x / LANES;
    if (i < v.n) ell_fetch<T, KF>(v.f_ell_col, v.f_ell_val, i, jc, sc);
    for (; i < v.n; i += ng) {
        const int64_t inext = i + ng;
        int jn[KF];
        T sn[KF];
        if (inext < v.n) ell_fetch<T, KF>(v.f_ell_col, v.f_ell_val, inext, jn, sn);
        const V ri = mask_tail(load_row(R, i, ldr, gl, active), gl * W, r);
        const T dsi = v.d_s[i];
        const T dlo = v.d_s_lo ? v.d_s_lo[i] : T(0);
        V gold = vzero(T()), dold = vzero(T());
        if (MODE == 1 && active) {
            gold = ld(G + i * ldr + gl * W);
            dold = ld(D + i * ldr + gl * W);
        }
        V gth[KF];
#pragma unroll
        for (int k = 0; k < KF; ++k) gth[k] = load_row(R, jc[k], ldr, gl, active);
        using Acc = typename AccOf<T>::type;
        Acc acc;
        acc.init();
        acc.add(dsi, ri);
        if (sizeof(T) == 4) acc.add_lo(dlo, ri);
#pragma unroll
        for (int k = 0; k < KF; ++k) acc.add(sc[k], gth[k]);
        const V g = mask_tail(scale4(T(2), acc.value()), gl * W, r);
        pgg = dot_add(g, g, pgg);
        if (MODE == 1) {
            V z = g;
            if (pc && sizeof(T) == 8 && v.pc_rec) {  // the row's divisions come with its slack diagonal
                const T rg = group_sum<LANES>(dot(ri, g), gmask);
                const double2 q = v.pc_rec[i];
                z = scale4(T(q.x), fma4(T(-q.y) * rg, ri, g));
            } else if (pc) {
                const T rg = group_sum<LANES>(dot(ri, g), gmask), rr = group_sum<LANES>(dot(ri, ri), gmask);
                T sdi = dsi + dlo;
                sdi = sdi > pc_floor ? sdi : pc_floor;
                const int k = v.d_sel_k[i];
                const T a = k >= 0 ? T(v.d_sel_a[i]) : T(0);
                const T ka = T(4) * sig * a * a;
                const T coef = ka * rg / (T(2) * sdi + ka * rr);
                z = scale4(T(1) / (T(2) * sdi), fma4(-coef, ri, g));
            }
            pzg = dot_add(z, g, pzg);
            pgo = dot_add(g, gold, pgo);
            pgd = dot_add(g, dold, pgd);
            if (writer) stv(G + i * ldr + gl * W, z);
        } else if (writer) {
            stv(G + i * ldr + gl * W, g);
        }
#pragma unroll
        for (int k = 0; k < KF; ++k) {
            jc[k] = jn[k];
            sc[k] = sn[k];
        }
    }
    double *part = partials + size_t(blockIdx.x) * kPartStride;
    const double vals[4] = {double(pgg), double(pgo), double(pgd), double(pzg)};
    block_partials<4>(vals, part, shm);
    if (!last_block(&st->counter[CNT_SPMM])) return;
    double tot[4];
    sum_partials_n<4>(partials, tot, shm);
    if (threadIdx.x == 0) {
        if (MODE == 1) {
            spmm_finish(st, tot[0], tot[1], tot[2], tot[3]);
        } else {
            st->gg = tot[0];
            if (res) {
                res->gg = tot[0];
                __threadfence_system();
            }
        }
    }
}


// D = -G + beta D
template <typename T>
__global__ void __launch_bounds__(kBlock) k_dir(const T *__restrict__ G, T *__restrict__ D, int64_t nvec,
                                                const DevState *st, const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    const T beta = T(st->beta);
    const V *g = reinterpret_cast<const V *>(G);
    V *d = reinterpret_cast<V *>(D);
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < nvec; t += int64_t(gridDim.x) * blockDim.x) {
        const V gv = g[t];
        V dv = (beta != T(0)) ? d[t] : vzero(T());  // D may hold stale values when beta = 0
        d[t] = fma4(beta, dv, scale4(T(-1), gv));
    }
}


// ---------------------------------------------------------------------------------------
// (c) exact line search along D.  With a1 = A(RD^T + DR^T), a2 = A(DD^T) and S = C - A^*(w)
// at the current R, phi(alpha) = L(R + alpha D) has
//   q1 = <S, RD^T + DR^T> (= <grad_R L, D>),  q2 = <S, DD^T> + sigma/2 |a1|^2,
//   q3 = sigma a1.a2,  q4 = sigma/2 |a2|^2,  q0 = L
// (the expansion of Eq. AL with c_k - w.a_k folded into <S, .>).
//   MODE 0: coefficients and step only.
//   MODE 1: inner loop: q1 from the SpMM's inner products (<G, D> = -|G|^2 + beta <G, D_old>,
//           free of cancellation), plus the done / iteration bookkeeping.
// ---------------------------------------------------------------------------------------
template <typename T, int LANES, int SP, bool OFFSEL, bool LR, int MODE>
__global__ void __launch_bounds__(kBlock, 3) k_ls(SparseView<T> v, const T *__restrict__ R, const T *__restrict__ D,
                                               int r, int ldr, HostResult *res, DevState *st, double *partials,
                                               const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    constexpr int GW = LANES * SP;
    constexpr int U = 2;  // entries per subgroup and round (each gathers a row of R and one of D)
    __shared__ double shm[32 * 32];
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LANES - 1), sub = (lane & (GW - 1)) / LANES;
    const unsigned gmask = group_mask<GW>(lane);
    const int64_t g0 = int64_t(blockIdx.x) * (kBlock / GW) + threadIdx.x / GW;
    const int64_t ng = int64_t(gridDim.x) * (kBlock / GW);
    const bool active = gl * W < r;
    T p1 = T(0), p2 = T(0), p11 = T(0), p12 = T(0), p22 = T(0);
    auto sel_terms = [&](int k, T a, T x1, T x2) {
        if (k >= 0) {
            const T A1 = a * x1, A2 = a * x2;
            p11 += A1 * A1;
            p12 += A1 * A2;
            p22 += A2 * A2;
        }
    };
    // strict upper entries e0 .. e1-1 of a row: <S, RD^T + DR^T> and <S, DD^T> are lane-local
    // sums over the lane's columns; only an entry's selector needs its whole dot products
    auto upper = [&](V ri, V di, int64_t i, int e0, int e1) {
        for (int e = e0 + sub; e < e1 + sub; e += U * SP) {  // group-uniform trip count
            int j[U];
            T s2[U];
            V rj[U], dj[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const bool in = e + k * SP < e1;
                j[k] = in ? v.up_col[e + k * SP] : int(i);
                s2[k] = in ? T(2) * v.up_s[e + k * SP] : T(0);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                rj[k] = load_row(R, j[k], ldr, gl, active);
                dj[k] = load_row(D, j[k], ldr, gl, active);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                T x1 = dot(ri, dj[k]) + dot(di, rj[k]);
                T x2 = dot(di, dj[k]);
                p1 += s2[k] * x1;
                p2 += s2[k] * x2;
                if (OFFSEL) {
                    x1 = group_sum<LANES>(x1, gmask);
                    x2 = group_sum<LANES>(x2, gmask);
                    if (gl == 0 && e + k * SP < e1) sel_terms(v.up_sel_k[e + k * SP], v.up_sel_a2[e + k * SP], x1, x2);
                }
            }
        }
    };
    for (int64_t i = g0; i < v.n; i += ng) {
        const V ri = mask_tail(load_row(R, i, ldr, gl, active), gl * W, r);
        const V di = mask_tail(load_row(D, i, ldr, gl, active), gl * W, r);
        const int e0 = v.up_ptr[i], e1 = min(v.up_ptr[i + 1], e0 + kUpSeg);
        const T rdi = T(2) * dot(ri, di), ddi = dot(di, di);
        if (sub == 0) {
            const T si = v.d_s[i];
            p1 += si * rdi;
            p2 += si * ddi;
        }
        const int ksel = v.d_sel_k[i];
        if (ksel >= 0) {  // group-uniform
            const T a1 = group_sum<LANES>(rdi, gmask);
            const T a2 = group_sum<LANES>(ddi, gmask);
            if (gl == 0 && sub == 0) sel_terms(ksel, sizeof(T) == 4 ? T(v.d_sel_af[i]) : T(v.d_sel_a[i]), a1, a2);
        }
        upper(ri, di, i, e0, e1);
    }
    for (int64_t q = g0; q < v.n_useg; q += ng) {  // the rest of the long rows
        const int i = v.us_row[q], e0 = v.us_e0[q], e1 = min(v.up_ptr[i + 1], e0 + kUpSeg);
        upper(mask_tail(load_row(R, i, ldr, gl, active), gl * W, r),
              mask_tail(load_row(D, i, ldr, gl, active), gl * W, r), i, e0, e1);
    }
    double *part = partials + size_t(blockIdx.x) * kPartStride;
    const double vals[5] = {double(p1), double(p2), double(p11), double(p12), double(p22)};
    block_partials<5>(vals, part, shm);
    if (LR) block_lr_cols<T, LANES>(v, D, r, ldr, part + 8, shm);
    if (!last_block(&st->counter[CNT_LS])) return;
    double tot[5];
    sum_partials_n<5>(partials, tot, shm);
    if (LR) sum_lr_cols(partials + 8, v.lr_k, r, st->zd);
    if (v.m_gen > 0) {
        double g11 = 0.0, g12 = 0.0, g22 = 0.0;
        for (int g = threadIdx.x; g < v.m_gen; g += blockDim.x) {
            const double A1 = v.g_a1[g], A2 = v.g_a2[g];
            g11 += A1 * A1;
            g12 += A1 * A2;
            g22 += A2 * A2;
        }
        tot[2] += block_sum(g11, shm);
        tot[3] += block_sum(g12, shm);
        tot[4] += block_sum(g22, shm);
    }
    if (threadIdx.x == 0) {
        ls_finish<T, MODE, LR>(v, st, r, tot);
        if (res) ls_result(res, st);
    }
}

// ELL form of the line-search SDDMM (static S_off: no off-diagonal selector constraints,
// no low-rank C): one row per group and iteration, the next row's upper neighbours fetched
// ahead of the current row's gathers of R and D
template <typename T, int LANES, int KU, int MODE>
__global__ void __launch_bounds__(kBlock, 4) k_ls_ell(SparseView<T> v, const T *__restrict__ R,
                                                   const T *__restrict__ D, int r, int ldr, HostResult *res,
                                                   DevState *st, double *partials, const int *done) {
    if (*done) return;
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    __shared__ double shm[64];
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LANES - 1);
    const unsigned gmask = group_mask<LANES>(lane);
    const int gpb = kBlock / LANES;
    const int64_t ng = int64_t(gridDim.x) * gpb;
    const bool active = gl * W < r;
    T p1 = T(0), p2 = T(0), p11 = T(0), p12 = T(0), p22 = T(0);
    int jc[KU];
    T sc[KU];
    auto fetch = [&](int64_t row, int (&jj)[KU], T (&ss)[KU]) {
        if constexpr (KU == 2) ell_fetch2<T, KU>(v.u_ell_col, v.u_ell_val, row, jj, ss);
        else ell_fetch<T, KU>(v.u_ell_col, v.u_ell_val, row, jj, ss);
    };
    int64_t i = int64_t(blockIdx.x) * gpb + threadIdx.x / LANES;
    if (i < v.n) fetch(i, jc, sc);
    for (; i < v.n; i += ng) {
        const V ri = mask_tail(load_row(R, i, ldr, gl, active), gl * W, r);
        const V di = mask_tail(load_row(D, i, ldr, gl, active), gl * W, r);
        V rj[KU], dj[KU];
#pragma unroll
        for (int k = 0; k < KU; ++k) {
            rj[k] = load_row(R, jc[k], ldr, gl, active);
            dj[k] = load_row(D, jc[k], ldr, gl, active);
        }
        T sq[KU];
#pragma unroll
        for (int k = 0; k < KU; ++k) sq[k] = T(2) * sc[k];
        // the next row's neighbours, fetched while this row's gathers are in flight
        if (i + ng < v.n) fetch(i + ng, jc, sc);
        // <S, RD^T + DR^T> and <S, DD^T> need no per-row reduction: every lane accumulates its
        // columns' share (the S values are the same for all lanes of the row) and the block
        // reduction at the end sums lanes and rows together.  Only the diagonal selector's
        // a1, a2 are reduced per row (their squares enter q2..q4).
        const T rdi = dot(ri, di), ddi = dot(di, di);
        const T sii = v.d_s[i];
        T l1 = T(2) * sii * rdi, l2 = sii * ddi;
#pragma unroll
        for (int k = 0; k < KU; ++k) {
            l1 += sq[k] * (dot(ri, dj[k]) + dot(di, rj[k]));
            l2 += sq[k] * dot(di, dj[k]);
        }
        p1 += l1;
        p2 += l2;
        const int ksel = v.d_sel_k[i];
        if (ksel >= 0) {  // group-uniform
            const T a1 = T(2) * group_sum<LANES>(rdi, gmask);
            const T a2 = group_sum<LANES>(ddi, gmask);
            if (gl == 0) {
                const T a = T(v.d_sel_a[i]);
                const T A1 = a * a1, A2 = a * a2;
                p11 += A1 * A1;
                p12 += A1 * A2;
                p22 += A2 * A2;
            }
        }
    }
    const double vals[5] = {double(p1), double(p2), double(p11), double(p12), double(p22)};
    block_partials<5>(vals, partials + size_t(blockIdx.x) * kPartStride, shm);
    if (!last_block(&st->counter[CNT_LS])) return;
    double tot[5];
    sum_partials_n<5>(partials, tot, shm);
    if (threadIdx.x == 0) {
        ls_finish<T, MODE, false>(v, st, r, tot);
        if (res) ls_result(res, st);
    }
}


// R += alpha D  (skipped when done == 1; done == 2, the step that reached the iteration cap,
// still takes this update and then becomes done == 1, so that the remaining launches of the
// chunk apply nothing)
template <typename T>
__global__ void __launch_bounds__(kBlock) k_axpy(T *__restrict__ R, const T *__restrict__ D, int64_t nvec,
                                                 DevState *st, const int *done, int final_only) {
    const int d = *done;
    if (d == 1 || (final_only && d != 2)) return;
    using V = typename VecT<T>::type;
    const T alpha = T(st->alpha);
    V *x = reinterpret_cast<V *>(R);
    const V *dv = reinterpret_cast<const V *>(D);
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < nvec; t += int64_t(gridDim.x) * blockDim.x)
        x[t] = fma4(alpha, dv[t], x[t]);
    if (d == 2 && last_block(&st->counter[CNT_AXPY]) && threadIdx.x == 0) st->done = 1;
}

// dst (n x ld_dst) <- src (n x ld_src) columns 0..r-1, zero columns r..ld_dst-1,
// optionally column r <- scale * col
template <typename T>
__global__ void __launch_bounds__(kBlock) k_relayout(const T *__restrict__ src, int ld_src, T *__restrict__ dst,
                                                     int ld_dst, int r, int64_t n, const T *__restrict__ col,
                                                     double scale) {
    const int64_t total = n * ld_dst;
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < total; t += int64_t(gridDim.x) * blockDim.x) {
        const int64_t i = t / ld_dst;
        const int c = int(t - i * ld_dst);
        T x = T(0);
        if (c < r) x = src[i * ld_src + c];
        else if (c == r && col) x = T(scale * double(col[i]));
        dst[t] = x;
    }
}

// st->red[0] = sum_k x_k^2
static __global__ void __launch_bounds__(kBlock) k_sumsq(const double *__restrict__ x, int64_t m, DevState *st,
                                                  double *partials) {
    __shared__ double shm[64];
    double acc = 0.0;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < m; k += int64_t(gridDim.x) * blockDim.x)
        acc += x[k] * x[k];
    const double t = block_sum(acc, shm);
    if (threadIdx.x == 0) partials[size_t(blockIdx.x) * kPartStride] = t;
    if (!last_block(&st->counter[CNT_RED])) return;
    const double s = sum_partials(partials, 0, shm);
    if (threadIdx.x == 0) st->red[0] = s;
}

// ---------------------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------------------

// Subgroups per row, a warp's worth or one: splitting a row costs a merge of the subgroups' sums (in
// FP64 up to ten additions), so it pays where the walk is long (the rows' mean length as an entry sees
// it, f_len and up_len, so that the long rows of a heavy-tailed graph count for what they hold), or
// where one subgroup a row leaves most of the chip idle.  The lines below give close to the smallest
// loss against the better of the two over ER graphs of 400 to 60,000 rows and degree 4 to 320, Kronecker
// graphs, theta and matrix completion problems, r = 1 to 32 (1,244 cells; at worst 1.25 of the better).
// k_spmm: eight entries a subgroup, or half an entry below 152 x 128 lanes of rows.  us of alm_grad, one /
// a warp's worth: ER(60,000) of degree 24, r = 1, FP64 61 / 147, r = 13, FP32 74 / 91; of degree 36,
// r = 32, FP32 113 / 126; Kronecker of 2^16 rows, r = 8, FP32 139 / 110, FP64 215 / 178.
template <typename T>
static inline bool wide_spmm(const LaunchCtx &c, const SparseView<T> &v, int LN) {
    return v.f_len >= 8 * (32 / LN) ||
           (int64_t(v.n) * LN < int64_t(c.sms) * 128 && 4 * v.nnz_u >= (32 / LN) * int64_t(v.n));
}
// k_ls (two gathers an entry, a merge of scalars only) and k_inner_off: two entries, three where the rows
// fill the chip several times over, one with off-diagonal selectors (whose dot products are summed over
// the row group entry by entry), or a quarter of an entry below 152 x 128 lanes.  us of
// alm_linesearch: ER(60,000) of degree 36, r = 1, FP64 156 / 214, of degree 24, r = 8, FP64 206 / 249;
// ER(2,000) of degree 48, r = 32, FP32 63 / 56; Kronecker of 2^16 rows, r = 1, FP64 384 / 248; theta SDP
// n = 5000, r = 8, FP64 141 / 126, n = 20,000, r = 1, FP64 140 / 158.
template <typename T>
static inline bool wide_ls(const LaunchCtx &c, const SparseView<T> &v, int LN) {
    const int64_t lanes = int64_t(v.n) * LN;
    const int need = v.has_off_sel ? 1 : lanes < int64_t(c.sms) * 1024 ? 2 : 3;
    return v.up_len >= need * (32 / LN) ||
           (lanes < int64_t(c.sms) * 128 && 4 * v.nnz_u >= (32 / LN) * int64_t(v.n));
}
#define ALM_ROW_SPLIT(wide, LN, ...)                                             \
    if (wide) { constexpr int SPW = 32 / LN; __VA_ARGS__; }                      \
    else { constexpr int SPW = 1; __VA_ARGS__; }

// Whether k_eval walks the upper entries by rows: FP32, at most two upper entries a row and a factor
// of 30 MB or more.  us a call, by rows / by entries: torus 449^2, r = 32 (26 MB) 65 / 64; 700^2,
// r = 16 (31 MB) 69 / 72, r = 32 94 / 110; 1000^2, r = 32 150 / 183; random 3-regular 1e6, r = 32
// 166 / 168; FP64, torus 700^2, r = 32 274 / 256.
template <typename T>
static inline bool eval_by_row(const SparseView<T> &v, int ldr) {
    return sizeof(T) == 4 && v.nnz_u <= 2 * int64_t(v.n) && int64_t(v.n) * ldr * 4 >= 30000000;
}
template <typename T, int LN, bool OFF, bool LRB, bool FUS>
static void eval_one(const LaunchCtx &c, const SparseView<T> &v, const T *R, int r, int ldr, double *AX,
                     const double *y, double *w, const int *done) {
    // rows per row group and round: up to one per lane (for the FP64 work of the rows), as
    // long as the rounds still give every multiprocessor 16 warps
    const int64_t rw = 32 / LN;
    const int nb = int(std::max<int64_t>(1, std::min<int64_t>(LN, v.n / (rw * 16 * c.sms))));
    if constexpr (sizeof(T) == 4 && !OFF) {
        if (eval_by_row(v, ldr)) {
            auto *fn = k_eval<T, LN, true, OFF, LRB, FUS>;
            const int grid = grid_for(c, fn, v.n + v.n_useg * nb, kBlock / LN * nb);
            fn<<<grid, kBlock, 0, c.stream>>>(v, R, r, ldr, AX, y, w, nb, c.sigma, c.res, c.st, c.partials, done);
            return;
        }
    }
    auto *fn = k_eval<T, LN, false, OFF, LRB, FUS>;
    int ge = v.diag_only ? 1 : grid_for(c, fn, v.nnz_u, 2 * (kBlock / LN));
    // every CTA has its reductions of the low-rank sums to do and to leave to the last one: from one CTA
    // a multiprocessor on, two rounds of entries a CTA (theta SDP n = 5000, r = 32, FP32: k_eval 33.6 -> 25.2 us)
    if (LRB && !v.diag_only) ge = std::max(std::min(ge, c.sms), grid_for(c, fn, v.nnz_u, 4 * (kBlock / LN)));
    const int grid = std::max(grid_for(c, fn, v.n, kBlock / LN * nb), ge);
    fn<<<grid, kBlock, 0, c.stream>>>(v, R, r, ldr, AX, y, w, nb, c.sigma, c.res, c.st, c.partials, done);
}

template <typename T>
void launch_eval(const LaunchCtx &c, const SparseView<T> &v, const T *R, int r, int ldr, double *AX, const int *done,
                 const double *y, double *w) {
    constexpr int W = VecT<T>::W;
    const int L = lanes_for(r, W);
    if (v.m_gen > 0) {
        ALM_DISPATCH_LANES(L, {
            k_gen<T, LN, false><<<std::min(v.n_gchunk, c.grid), kBlock, 0, c.stream>>>(v, R, R, r, ldr, AX, done);
        });
        ++*c.launches;
    }
    const bool fused = v.fused_dual && y && w;
    const bool off = v.has_off_sel, lr = v.lr_k > 0;
    ALM_DISPATCH_LANES(L, {
        if (fused) {
            if (lr) eval_one<T, LN, false, true, true>(c, v, R, r, ldr, AX, y, w, done);
            else eval_one<T, LN, false, false, true>(c, v, R, r, ldr, AX, y, w, done);
        } else if (off && lr) eval_one<T, LN, true, true, false>(c, v, R, r, ldr, AX, y, w, done);
        else if (off) eval_one<T, LN, true, false, false>(c, v, R, r, ldr, AX, y, w, done);
        else if (lr) eval_one<T, LN, false, true, false>(c, v, R, r, ldr, AX, y, w, done);
        else eval_one<T, LN, false, false, false>(c, v, R, r, ldr, AX, y, w, done);
    });
    ++*c.launches;
}

template <typename T>
void launch_inner_slack(const LaunchCtx &c, const SparseView<T> &v, T *R, const T *D, int r, int ldr,
                        const int *done) {
    constexpr int W = VecT<T>::W;
    const int L = lanes_for(r, W);
    if constexpr (sizeof(T) == 8) {
        ALM_DISPATCH_LANES(L, {
            auto *fn = D ? k_inner_slack64<LN, true> : k_inner_slack64<LN, false>;
            const int grid = grid_for(c, fn, v.n, kBlock);
            fn<<<grid, kBlock, 0, c.stream>>>(v, R, D, r, ldr, c.st, done);
        });
    } else {
        ALM_DISPATCH_LANES(L, {
            auto *fn = D ? k_inner_slack<T, LN, true> : k_inner_slack<T, LN, false>;
            const int grid = grid_for(c, fn, v.n, 4 * (kBlock / LN));
            fn<<<grid, kBlock, 0, c.stream>>>(v, R, D, r, ldr, c.st, done);
        });
    }
    ++*c.launches;
}

template <typename T>
void launch_inner_off(const LaunchCtx &c, const SparseView<T> &v, const T *R, int r, int ldr, const int *done) {
    const int L = lanes_for(r, VecT<T>::W);
    ALM_DISPATCH_LANES(L, {
        ALM_ROW_SPLIT(wide_ls(c, v, LN), LN, {
            auto *fn = k_inner_off<T, LN, SPW>;
            const int grid = grid_for(c, fn, v.n + v.n_useg, kBlock / (LN * SPW));
            fn<<<grid, kBlock, 0, c.stream>>>(v, R, r, ldr, c.st, done);
        });
    });
    ++*c.launches;
}

template <typename T>
void launch_prep_off(const LaunchCtx &c, const SparseView<T> &v, const double *y) {
    auto *fn = k_prep_off<T>;
    fn<<<grid_for(c, fn, v.nnz_u, kBlock * 4), kBlock, 0, c.stream>>>(v, y);
    ++*c.launches;
}

template <typename T>
void launch_prep_base(const LaunchCtx &c, const SparseView<T> &v, const double *y, T *base_hi, T *base_lo) {
    auto *fn = k_prep_base<T>;
    const int grid = grid_for(c, fn, v.n, kBlock * 4);
    fn<<<grid, kBlock, 0, c.stream>>>(v, y, base_hi, base_lo);
    ++*c.launches;
}

template <typename T>
void launch_dual_slack(const LaunchCtx &c, const SparseView<T> &v, const double *y, const double *AX, double *w,
                       const int *done, const int2 *up_slot) {
    int64_t items = v.n > v.m ? v.n : v.m;
    if (v.off_dynamic && v.nnz_u > items) items = v.nnz_u;
    auto *fn = k_dual_slack<T>;
    const int grid = grid_for(c, fn, items, kBlock * 2);
    fn<<<grid, kBlock, 0, c.stream>>>(v, y, AX, w, up_slot, c.st, c.partials, done);
    ++*c.launches;
}

template <typename T, int LN, bool LRB, int MODE>
static void spmm_one(const LaunchCtx &c, const SparseView<T> &v, const T *R, int r, int ldr, T *G, const T *D,
                     const int *done) {
    if (v.n_heavy > 0) {
        k_spmm_heavy<T, LN><<<std::min(v.n_hseg, c.grid), kBlock, 0, c.stream>>>(v, R, r, ldr, done);
        ++*c.launches;
    }
    ALM_ROW_SPLIT(wide_spmm(c, v, LN), LN, {
        auto *fn = k_spmm<T, LN, SPW, LRB, MODE>;
        const int grid = grid_for(c, fn, v.n, kBlock / (LN * SPW));
        fn<<<grid, kBlock, 0, c.stream>>>(v, R, r, ldr, G, D, c.res, c.st, c.partials, done);
    });
}

template <typename T, int LN, int KF>
static void spmm_ell_one(const LaunchCtx &c, const SparseView<T> &v, const T *R, int r, int ldr, T *G, const T *D,
                         int mode, const int *done) {
    if (mode == 1) {
        auto *fn = k_spmm_ell<T, LN, KF, 1>;
        fn<<<grid_for(c, fn, v.n, kBlock / LN), kBlock, 0, c.stream>>>(v, R, r, ldr, G, D, c.res, c.st, c.partials,
                                                                             done);
    } else {
        auto *fn = k_spmm_ell<T, LN, KF, 0>;
        fn<<<grid_for(c, fn, v.n, kBlock / LN), kBlock, 0, c.stream>>>(v, R, r, ldr, G, D, c.res, c.st, c.partials,
                                                                             done);
    }
}

template <typename T>
void launch_spmm(const LaunchCtx &c, const SparseView<T> &v, const T *R, int r, int ldr, T *G, const T *D, int mode,
                 const int *done) {
    constexpr int W = VecT<T>::W;
    const int L = lanes_for(r, W);
    const bool lr = v.lr_k > 0;
    if (v.ell_kf > 0 && !lr) {
        ALM_DISPATCH_LANES(L, {
            if (v.ell_kf == 4) spmm_ell_one<T, LN, 4>(c, v, R, r, ldr, G, D, mode, done);
            else if (v.ell_kf == 8) spmm_ell_one<T, LN, 8>(c, v, R, r, ldr, G, D, mode, done);
            else spmm_ell_one<T, LN, 16>(c, v, R, r, ldr, G, D, mode, done);
        });
        ++*c.launches;
        return;
    }
    ALM_DISPATCH_LANES(L, {
        if (mode == 1) {
            if (lr) spmm_one<T, LN, true, 1>(c, v, R, r, ldr, G, D, done);
            else spmm_one<T, LN, false, 1>(c, v, R, r, ldr, G, D, done);
        } else {
            if (lr) spmm_one<T, LN, true, 0>(c, v, R, r, ldr, G, D, done);
            else spmm_one<T, LN, false, 0>(c, v, R, r, ldr, G, D, done);
        }
    });
    ++*c.launches;
}

template <typename T>
void launch_dir(const LaunchCtx &c, const T *G, T *D, int64_t count, const int *done) {
    constexpr int W = VecT<T>::W;
    const int64_t nvec = count / W;
    auto *fn = k_dir<T>;
    const int grid = grid_for(c, fn, nvec, kBlock * 2);
    fn<<<grid, kBlock, 0, c.stream>>>(G, D, nvec, c.st, done);
    ++*c.launches;
}

template <typename T, int LN, bool OFF, bool LRB, int MODE>
static void ls_one(const LaunchCtx &c, const SparseView<T> &v, const T *R, const T *D, int r, int ldr,
                   const int *done) {
    ALM_ROW_SPLIT(wide_ls(c, v, LN), LN, {
        auto *fn = k_ls<T, LN, SPW, OFF, LRB, MODE>;
        const int grid = grid_for(c, fn, v.n + v.n_useg, kBlock / (LN * SPW));
        fn<<<grid, kBlock, 0, c.stream>>>(v, R, D, r, ldr, c.res, c.st, c.partials, done);
    });
}

template <typename T, int LN, int KU>
static void ls_ell_one(const LaunchCtx &c, const SparseView<T> &v, const T *R, const T *D, int r, int ldr, int mode,
                       const int *done) {
    if (mode == 1) {
        auto *fn = k_ls_ell<T, LN, KU, 1>;
        fn<<<grid_for(c, fn, v.n, kBlock / LN), kBlock, 0, c.stream>>>(v, R, D, r, ldr, c.res, c.st, c.partials, done);
    } else {
        auto *fn = k_ls_ell<T, LN, KU, 0>;
        fn<<<grid_for(c, fn, v.n, kBlock / LN), kBlock, 0, c.stream>>>(v, R, D, r, ldr, c.res, c.st, c.partials, done);
    }
}

template <typename T>
void launch_ls(const LaunchCtx &c, const SparseView<T> &v, const T *R, const T *D, int r, int ldr, const double *w,
               int mode, const int *done) {
    (void)w;
    constexpr int W = VecT<T>::W;
    const int L = lanes_for(r, W);
    if (v.ell_ku > 0 && v.lr_k == 0 && !v.has_off_sel && v.m_gen == 0) {
        ALM_DISPATCH_LANES(L, {
            if (v.ell_ku == 2) ls_ell_one<T, LN, 2>(c, v, R, D, r, ldr, mode, done);
            else if (v.ell_ku == 4) ls_ell_one<T, LN, 4>(c, v, R, D, r, ldr, mode, done);
            else if (v.ell_ku == 8) ls_ell_one<T, LN, 8>(c, v, R, D, r, ldr, mode, done);
            else ls_ell_one<T, LN, 16>(c, v, R, D, r, ldr, mode, done);
        });
        ++*c.launches;
        return;
    }
    if (v.m_gen > 0) {
        ALM_DISPATCH_LANES(L, {
            k_gen<T, LN, true><<<std::min(v.n_gchunk, c.grid), kBlock, 0, c.stream>>>(v, R, D, r, ldr, nullptr, done);
        });
        ++*c.launches;
    }
    const bool off = v.has_off_sel, lr = v.lr_k > 0;
#define ALM_LS(OFF, LRB)                                                     \
    if (mode == 1) ls_one<T, LN, OFF, LRB, 1>(c, v, R, D, r, ldr, done);    \
    else ls_one<T, LN, OFF, LRB, 0>(c, v, R, D, r, ldr, done);
    ALM_DISPATCH_LANES(L, {
        if (off && lr) { ALM_LS(true, true) }
        else if (off) { ALM_LS(true, false) }
        else if (lr) { ALM_LS(false, true) }
        else { ALM_LS(false, false) }
    });
#undef ALM_LS
    ++*c.launches;
}

template <typename T>
void launch_axpy(const LaunchCtx &c, T *R, const T *D, int64_t count, const int *done, int final_only) {
    constexpr int W = VecT<T>::W;
    const int64_t nvec = count / W;
    auto *fn = k_axpy<T>;
    const int grid = grid_for(c, fn, nvec, kBlock * 2);
    fn<<<grid, kBlock, 0, c.stream>>>(R, D, nvec, c.st, done, final_only);
    ++*c.launches;
}

// the same with 16-byte rows parts: no appended column, row strides a multiple of the vector
// (checked by every caller of the API; 1e6 rows x 32 floats 77 -> 36 us)
template <typename T>
__global__ void __launch_bounds__(kBlock) k_relayout_vec(const T *__restrict__ src, int ld_src, T *__restrict__ dst,
                                                         int ld_dst, int r, int64_t n) {
    using V = typename VecT<T>::type;
    constexpr int W = VecT<T>::W;
    const unsigned per = unsigned(ld_dst / W);
    for (int64_t i = int64_t(blockIdx.x) * (kBlock / 8) + threadIdx.x / 8; i < n; i += int64_t(gridDim.x) * (kBlock / 8))
        for (unsigned q = threadIdx.x % 8; q < per; q += 8) {
            const int c = int(q) * W;
            stv(dst + i * ld_dst + c, c < r ? mask_tail(ldro(src + i * ld_src + c), c, r) : vzero(T()));
        }
}

template <typename T>
void launch_relayout(const LaunchCtx &c, const T *src, int ld_src, T *dst, int ld_dst, int r, int64_t n, const T *col,
                     double scale) {
    constexpr int W = VecT<T>::W;
    if (!col && ld_src % W == 0 && ld_dst % W == 0) {
        auto *fv = k_relayout_vec<T>;
        fv<<<grid_for(c, fv, n, kBlock / 8), kBlock, 0, c.stream>>>(src, ld_src, dst, ld_dst, r, n);
        ++*c.launches;
        return;
    }
    auto *fn = k_relayout<T>;
    const int grid = grid_for(c, fn, n * ld_dst, kBlock * 4);
    fn<<<grid, kBlock, 0, c.stream>>>(src, ld_src, dst, ld_dst, r, n, col, scale);
    ++*c.launches;
}

template <typename T>
void launch_sumsq(const LaunchCtx &c, const double *x, int64_t m) {
    const int grid = grid_for(c, k_sumsq, m, kBlock * 4);
    k_sumsq<<<grid, kBlock, 0, c.stream>>>(x, m, c.st, c.partials);
    ++*c.launches;
}

#define ALM_INST(T)                                                                                              \
    template void launch_eval<T>(const LaunchCtx &, const SparseView<T> &, const T *, int, int, double *,        \
                                 const int *, const double *, double *);                                         \
    template void launch_dual_slack<T>(const LaunchCtx &, const SparseView<T> &, const double *, const double *, \
                                       double *, const int *, const int2 *);                                     \
    template void launch_inner_slack<T>(const LaunchCtx &, const SparseView<T> &, T *, const T *, int, int,      \
                                        const int *);                                                             \
    template void launch_inner_off<T>(const LaunchCtx &, const SparseView<T> &, const T *, int, int, const int *); \
    template void launch_prep_off<T>(const LaunchCtx &, const SparseView<T> &, const double *);                  \
    template void launch_prep_base<T>(const LaunchCtx &, const SparseView<T> &, const double *, T *, T *);      \
    template void launch_spmm<T>(const LaunchCtx &, const SparseView<T> &, const T *, int, int, T *, const T *,  \
                                 int, const int *);                                                              \
    template void launch_dir<T>(const LaunchCtx &, const T *, T *, int64_t, const int *);                         \
    template void launch_ls<T>(const LaunchCtx &, const SparseView<T> &, const T *, const T *, int, int,         \
                               const double *, int, const int *);                                                \
    template void launch_axpy<T>(const LaunchCtx &, T *, const T *, int64_t, const int *, int);                   \
    template void launch_relayout<T>(const LaunchCtx &, const T *, int, T *, int, int, int64_t, const T *,       \
                                     double);                                                                    \
    template void launch_sumsq<T>(const LaunchCtx &, const double *, int64_t);

// ALM_INST_ONLY (1: float, 2: double) lets the build compile the two precisions as separate
// objects in parallel
#if !defined(ALM_INST_ONLY) || ALM_INST_ONLY == 1
ALM_INST(float)
#endif
#if !defined(ALM_INST_ONLY) || ALM_INST_ONLY == 2
ALM_INST(double)
#endif

}  // namespace alm
