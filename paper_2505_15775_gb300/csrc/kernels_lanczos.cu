// Lanczos kernels for the smallest eigenpair of S = C - A^*(w) = grad_X L_sigma
// (arXiv 2505.15775, Alg. 1: eigenvectors of grad_X L drive the rank growth;
// Sec. 6: lambda_min(C - A^* y) is the dual term of the KKT error)  [hot path (d)].
//
// One restart cycle builds an orthonormal basis Q = [q_0 .. q_m] (column-major,
// each q_l contiguous) of the Krylov space of S.  Step j (three launches; four with a low-rank
// part of C, whose products u_l^T q need the normalised vector):
//   k_lz_reorth<SPMV>  q_j = w / beta_{j-1}, w = S q_j (sparse part, diagonal, low-rank part of
//                      C), formed in registers and stored, then h1 = Q^T w
//   k_lz_reorth x2     the rest of classical Gram-Schmidt against q_0..q_j, applied twice:
//                      w -= Q h1; h2 = Q^T w; w -= Q h2; beta_j = ||w||
//                      (alpha_j = h1_j + h2_j)
//   k_lz_normalize     q_{j+1} = w / beta_j (only with a low-rank part)
// (k_lz_spmv alone serves the residual check of the final Ritz pair)
// and at the end of a cycle
//   k_lz_tridiag    smallest eigenpair (theta, s) of the m x m tridiagonal T in FP64
//                   (tridiag.cuh), residual estimate |beta_{m-1} s_{m-1}|
//   k_lz_ritz       v = Q s, the next start vector / the result.
// Vectors are stored in the working precision; dot products sum in it within a warp and in FP64
// across warps, the start vector's norm in FP64 throughout.
//
// Short vectors (lz_cluster_rows) take k_lz_cluster instead: the whole eigensolve, start
// vector to residual, in one launch of one thread-block cluster.
#include <cooperative_groups.h>

#include <cfloat>
#include <cmath>
#include <mutex>

#include "dev_util.cuh"
#include "tridiag.cuh"

namespace alm {

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014) as a counter-based generator:
// element i of the stream `seed` is mix(seed + (i + 1) * golden_gamma).
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t i) {
    uint64_t z = seed + (i + 1) * 0x9e3779b97f4a7c15ULL;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_lz_start(T *__restrict__ q, int64_t n, uint64_t seed, DevState *st,
                                                     double *partials) {
    __shared__ double shm[32];
    double acc = 0.0;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const uint64_t z = splitmix64_at(seed, uint64_t(i));
        const double u = double(z >> 11) * (1.0 / 9007199254740992.0);  // [0, 1)
        const T x = T(2.0 * u - 1.0);
        q[i] = x;
        acc += double(x) * double(x);
    }
    const double t = block_sum(acc, shm);
    if (threadIdx.x == 0) partials[size_t(blockIdx.x) * kPartStride] = t;
    if (!last_block(&st->counter[CNT_LZ])) return;
    const double s = sum_partials(partials, 0, shm);
    if (threadIdx.x == 0) {
        st->nrm2 = s;
        st->lz_stop = 0;
        st->lz_m = 0;
        st->anorm = 0.0;
    }
}

// warm start: q += (0.05 / |u|) u (|u|^2 in st->nrm2 from k_lz_start), then |q|^2 -> st->nrm2
template <typename T>
__global__ void __launch_bounds__(kBlock) k_lz_mix(T *__restrict__ q, const T *__restrict__ u, int64_t n, DevState *st,
                                                   double *partials) {
    __shared__ double shm[32];
    const T sc = T(0.05 / sqrt(st->nrm2));
    double acc = 0.0;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const T x = q[i] + sc * u[i];
        q[i] = x;
        acc += double(x) * double(x);
    }
    const double t = block_sum(acc, shm);
    __syncthreads();  // every thread has read st->nrm2
    if (threadIdx.x == 0) partials[size_t(blockIdx.x) * kPartStride] = t;
    if (!last_block(&st->counter[CNT_LZ])) return;
    const double s = sum_partials(partials, 0, shm);
    if (threadIdx.x == 0) st->nrm2 = s;
}

// w = S q (one thread per row)
template <typename T>
__global__ void __launch_bounds__(kBlock) k_lz_spmv(SparseView<T> v, const T *__restrict__ q, T *__restrict__ w,
                                                    const DevState *st) {
    if (st->lz_stop) return;
    T qu[kMaxLR];
    for (int l = 0; l < v.lr_k; ++l) qu[l] = T(v.lr_s[l] * st->qu[l]);
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < v.n; i += int64_t(gridDim.x) * blockDim.x) {
        T acc = v.d_s[i] * q[i];
        const int e1 = v.f_ptr[i + 1];
        for (int e = v.f_ptr[i]; e < e1; ++e) acc += v.f_val[e] * q[v.f_col[e]];
        for (int l = 0; l < v.lr_k; ++l) acc += T(v.lr_u[int64_t(l) * v.n + i]) * qu[l];
        w[i] = acc;
    }
}

// stage 0: h = Q^T w, ||w||^2                      (j-th step, nvec = j + 1 basis vectors)
// stage 1: w -= Q h_in; h = Q^T w, ||w||^2
// stage 2: w -= Q h_in; ||w||^2 -> beta_j
// Rows are processed in tiles of kBlock * RPT (each thread keeps RPT entries of w in
// registers); products and per-warp sums are in the working precision, the per-warp
// sums are accumulated over tiles in FP64 in shared memory.
// SPMV (stage 0 only): the SpMV of the step is fused in -- each thread forms its rows of
// w = S q (as k_lz_spmv, same order of operations), stores them and keeps them in
// registers for the dot products, so w is not read back and the step has one launch less.
// With src the normalisation of the step before is fused in too: q = src / beta_{j-1} is formed
// where it is read (one product, as k_lz_normalize stores it) and the rows' owner stores it as
// basis column j; w then goes to the other buffer, as neighbours still read src.
//
// Bound: with 1 MB vectors and a basis in L2 the passes are latency, one warp's chain over the
// basis vectors.  Hence kLzUnroll vectors at a time: their loads are in flight together, and
// their warp sums share the shuffles -- in the first three rounds of the butterfly each lane
// keeps half of its vectors and hands over the other half, so eight vectors take 9 shuffles
// instead of 40, each sum over the same tree (the bits are those of one sum at a time).
// Torus 501 x 501, FP32, alm_lambda_min over two cycles (three): 4.56 (6.64) -> 3.48 (5.09) ms with the
// fused normalisation and the tridiagonal solve of tridiag.cuh, runs within 0.5% of each other.
constexpr int kLzUnroll = 8;
template <typename T, int RPT, bool SPMV>
__global__ void __launch_bounds__(kBlock) k_lz_reorth(SparseView<T> v, const T *__restrict__ src, T *qj,
                                                      const T *Q, int64_t ldq, int nvec, T *__restrict__ w,
                                                      int64_t n, const double *__restrict__ h_in, double *h_out, int j,
                                                      int stage, DevState *st, double *partials) {
    if (st->lz_stop) return;
    T qu[kMaxLR];
    if constexpr (SPMV)
        for (int l = 0; l < v.lr_k; ++l) qu[l] = T(v.lr_s[l] * st->qu[l]);
    constexpr int NW = kBlock / 32;
    constexpr int K = kLzUnroll;
    __shared__ T hs[kLzMax + K];
    __shared__ double wsum[NW][kLzMax + 2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int l = threadIdx.x; l < kLzMax + K; l += blockDim.x) hs[l] = stage > 0 && l < nvec ? T(h_in[l]) : T(0);
    for (int t = threadIdx.x; t < NW * (kLzMax + 2); t += blockDim.x) (&wsum[0][0])[t] = 0.0;
    __syncthreads();
    // the scale of q = scale * src (src null: q is column j, normalised already)
    T scale = T(1);
    if constexpr (SPMV)
        if (src) {
            const double beta = st->lz_beta[j - 1];
            scale = T(beta > 0.0 ? 1.0 / beta : 0.0);
        }
    const T *qin = SPMV ? (src ? src : qj) : nullptr;
    const int64_t tile = int64_t(kBlock) * RPT;
    T nrm = T(0);
    for (int64_t base = int64_t(blockIdx.x) * tile; base < n; base += int64_t(gridDim.x) * tile) {
        T x[RPT], own[RPT];
        int64_t idx[RPT];
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            idx[k] = base + threadIdx.x + int64_t(k) * kBlock;
            own[k] = T(0);
            if constexpr (SPMV) {
                T acc = T(0);
                if (idx[k] < n) {
                    const int64_t i = idx[k];
                    own[k] = src ? qin[i] * scale : qin[i];
                    acc = v.d_s[i] * own[k];
                    const int e1 = v.f_ptr[i + 1];
                    for (int e = v.f_ptr[i]; e < e1; ++e) {
                        const T q = qin[v.f_col[e]];
                        acc += v.f_val[e] * (src ? q * scale : q);
                    }
                    for (int l = 0; l < v.lr_k; ++l) acc += T(v.lr_u[int64_t(l) * v.n + i]) * qu[l];
                    w[i] = acc;
                    if (src) qj[i] = own[k];
                }
                x[k] = acc;
            } else {
                x[k] = idx[k] < n ? w[idx[k]] : T(0);
            }
        }
        if (stage > 0) {
            for (int l0 = 0; l0 < nvec; l0 += K) {
                T q[K][RPT];
#pragma unroll
                for (int u = 0; u < K; ++u)
#pragma unroll
                    for (int k = 0; k < RPT; ++k)
                        q[u][k] = l0 + u < nvec && idx[k] < n ? Q[int64_t(l0 + u) * ldq + idx[k]] : T(0);
#pragma unroll
                for (int u = 0; u < K; ++u)
#pragma unroll
                    for (int k = 0; k < RPT; ++k) x[k] -= q[u][k] * hs[l0 + u];  // 0 past nvec
            }
#pragma unroll
            for (int k = 0; k < RPT; ++k)
                if (idx[k] < n) w[idx[k]] = x[k];
        }
        if (stage < 2) {
            for (int l0 = 0; l0 < nvec; l0 += K) {
                T a[K];
#pragma unroll
                for (int u = 0; u < K; ++u) {
                    const int l = l0 + u;
                    a[u] = T(0);
#pragma unroll
                    for (int k = 0; k < RPT; ++k) {
                        // column j itself is this thread's own value when it was formed here
                        T q = T(0);
                        if (l < nvec && idx[k] < n) q = SPMV && src && l == j ? own[k] : Q[int64_t(l) * ldq + idx[k]];
                        a[u] += q * x[k];
                    }
                }
                // lane bits 4, 3, 2 pick the vector that the lane ends up with
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool up = lane & 16;
                    const T give = up ? a[u] : a[u + 4], keep = up ? a[u + 4] : a[u];
                    a[u] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const bool up = lane & 8;
                    const T give = up ? a[u] : a[u + 2], keep = up ? a[u + 2] : a[u];
                    a[u] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
                }
                {
                    const bool up = lane & 4;
                    const T give = up ? a[0] : a[1], keep = up ? a[1] : a[0];
                    a[0] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
                }
                a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
                a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
                const int l = l0 + ((lane & 16) ? 4 : 0) + ((lane & 8) ? 2 : 0) + ((lane & 4) ? 1 : 0);
                if ((lane & 3) == 0 && l < nvec) wsum[warp][l] += double(a[0]);
            }
        }
#pragma unroll
        for (int k = 0; k < RPT; ++k) nrm += x[k] * x[k];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    if (lane == 0) wsum[warp][kLzMax + 1] = double(nrm);
    __syncthreads();
    double *part = partials + size_t(blockIdx.x) * kPartStride;
    const int nslots = stage < 2 ? nvec : 0;
    for (int t = threadIdx.x; t <= nslots; t += blockDim.x) {
        const int from = t == 0 ? kLzMax + 1 : t - 1;
        double sacc = 0.0;
        for (int ww = 0; ww < NW; ++ww) sacc += wsum[ww][from];
        part[t] = sacc;  // slot 0: ||w||^2, slot 1 + l: (Q^T w)_l
    }
    if (!last_block(&st->counter[CNT_LZ])) return;
    // the slots' sums over blocks: one warp per slot, lanes over the blocks in a fixed order
    // (deterministic), all slots at once instead of one block reduction after another
    __shared__ double tot[kLzMax + 2];
    for (int t = warp; t <= nslots; t += NW) {
        double a = 0.0;
#pragma unroll 8
        for (int b = lane; b < int(gridDim.x); b += 32) a += __ldcg(partials + size_t(b) * kPartStride + t);
        a = warp_sum(a);
        if (lane == 0) tot[t] = a;
    }
    __syncthreads();
    if (stage < 2)
        for (int l = threadIdx.x; l < nvec; l += blockDim.x) h_out[l] = tot[1 + l];
    const double nrm2 = tot[0];
    if (threadIdx.x == 0) {
        st->nrm2 = nrm2;
        if (stage == 0) st->lz_alpha[j] = tot[1 + j];
        if (stage == 1) st->lz_alpha[j] += tot[1 + j];
        if (stage == 2) {
            const double beta = sqrt(nrm2);
            st->lz_beta[j] = beta;
            const double bprev = j > 0 ? st->lz_beta[j - 1] : 0.0;
            st->anorm = fmax(st->anorm, fabs(st->lz_alpha[j]) + beta + bprev);
            st->lz_m = j + 1;
            if (!(beta > 1e-13 * st->anorm)) st->lz_stop = 1;  // invariant subspace (or non-finite)
        }
    }
}

// mode 0: dst = src / sqrt(nrm2);   mode 1: dst = src / beta_j (skipped after a breakdown)
// both: qu_l = u_l^T dst
template <typename T>
__global__ void __launch_bounds__(kBlock) k_lz_normalize(SparseView<T> v, const T *__restrict__ src, T *__restrict__ dst,
                                                         int64_t n, int mode, int j, DevState *st, double *partials) {
    if (mode == 1 && st->lz_stop) return;
    __shared__ double shm[32];
    const double nrm = mode == 0 ? sqrt(st->nrm2) : st->lz_beta[j];
    const T sc = T(nrm > 0.0 ? 1.0 / nrm : 0.0);
    double acc[kMaxLR] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const T x = src[i] * sc;
        dst[i] = x;
        for (int l = 0; l < v.lr_k; ++l) acc[l] += v.lr_u[int64_t(l) * n + i] * double(x);
    }
    if (v.lr_k == 0) return;
    double *part = partials + size_t(blockIdx.x) * kPartStride;
    for (int l = 0; l < v.lr_k; ++l) {
        const double t = block_sum(acc[l], shm);
        if (threadIdx.x == 0) part[l] = t;
    }
    if (!last_block(&st->counter[CNT_LZ])) return;
    for (int l = 0; l < v.lr_k; ++l) {
        const double s = sum_partials(partials, l, shm);
        if (threadIdx.x == 0) st->qu[l] = s;
    }
}

// smallest eigenpair of the m x m tridiagonal T of the cycle (one warp)
__global__ void k_lz_tridiag(DevState *st, int mmax) {
    if (blockIdx.x != 0) return;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x >= 32) return;
    __shared__ double a[kLzMax], b[kLzMax];
    __shared__ int msh;
    if (lane == 0) msh = st->lz_m < mmax ? st->lz_m : mmax;
    __syncwarp();
    const int m = msh;
    if (m <= 0) return;
    for (int i = lane; i < m; i += 32) {
        a[i] = st->lz_alpha[i];
        b[i] = st->lz_beta[i];
    }
    __syncwarp();
    double resid = 0.0;
    const double theta = warp_tridiag_min(a, b, m, st->lz_s, &resid);
    if (lane != 0) return;
    st->theta = theta;
    st->resid_est = resid;
    st->lz_m = m;
}

// dst = Q[:, 0..m-1] s (and ||dst||^2)
template <typename T>
__global__ void __launch_bounds__(kBlock) k_lz_ritz(const T *__restrict__ Q, int64_t ldq, int mmax, T *__restrict__ dst,
                                                    int64_t n, DevState *st, double *partials) {
    __shared__ double shm[32];
    __shared__ double s[kLzMax];
    const int m = st->lz_m < mmax ? st->lz_m : mmax;
    for (int l = threadIdx.x; l < m; l += blockDim.x) s[l] = st->lz_s[l];
    __syncthreads();
    __shared__ T sT[kLzMax];
    for (int l = threadIdx.x; l < m; l += blockDim.x) sT[l] = T(s[l]);
    __syncthreads();
    T acc = T(0);
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        T x = T(0);
        for (int l = 0; l < m; ++l) x += Q[l * ldq + i] * sT[l];
        dst[i] = x;
        acc += x * x;
    }
    const double t = block_sum(double(acc), shm);
    if (threadIdx.x == 0) partials[size_t(blockIdx.x) * kPartStride] = t;
    if (!last_block(&st->counter[CNT_LZ])) return;
    const double nrm2 = sum_partials(partials, 0, shm);
    if (threadIdx.x == 0) st->nrm2 = nrm2;
}

// ||w - theta v||^2 -> st->red[1]   (true residual of the final Ritz pair)
template <typename T>
__global__ void __launch_bounds__(kBlock) k_lz_resid(const T *__restrict__ w, const T *__restrict__ v, int64_t n,
                                                     DevState *st, double *partials) {
    __shared__ double shm[32];
    const T th = T(st->theta);
    T acc = T(0);
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const T d = w[i] - th * v[i];
        acc += d * d;
    }
    const double t = block_sum(double(acc), shm);
    if (threadIdx.x == 0) partials[size_t(blockIdx.x) * kPartStride] = t;
    if (!last_block(&st->counter[CNT_LZ])) return;
    const double s = sum_partials(partials, 0, shm);
    if (threadIdx.x == 0) st->red[1] = s;
}

__global__ void k_lz_reset(DevState *st) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        st->lz_stop = 0;
        st->lz_m = 0;
    }
}

// ---------------------------------------------------------------------------------------
// The eigensolve of short vectors in one launch.  Four launches a step on vectors of 800
// entries are all latency: 60 us a step in FP64 (4 CTAs, serial walks over the basis, launch
// gaps), 32 steps and a tridiagonal solve a cycle.  Here one cluster of 16 CTAs runs every
// cycle: each CTA keeps its rows of the basis and of w in shared memory (row-major, one lane
// per basis vector, so that the dot products of a row with all vectors are one FMA
// instruction and need no shuffles), sums are exchanged through distributed shared memory, and
// the next Lanczos vector goes through global memory to every CTA's copy of q, which the SpMV
// gathers from.  A step is four cluster barriers (hardware, bounded): Q^T w, Q^T w again,
// |w|^2, the new q.  FP64 instructions are what is left (a warp's takes 64 cycles), so scalars
// are computed by one warp.  ER(800), FP64: 12 us a step, the tridiagonal solve's share included.
// ---------------------------------------------------------------------------------------
constexpr int kLzcThreads = 512, kLzcWarps = kLzcThreads / 32, kLzcMaxCtas = 16;
template <typename T>
struct LzcArgs {
    T *Q;                    // n x (k + 1), column-major; on return column 0 holds the Ritz vector
    int n, kk, pitch, nr;    // steps per cycle, pitch of a row's basis entries, rows per CTA
    int nv;                  // doubles per vector of partial sums
    int max_restarts, warm;
    double tol_rel, tol_abs;
    uint64_t seed;
};

template <typename T>
__global__ void __launch_bounds__(kLzcThreads, 1) k_lz_cluster(SparseView<T> v, LzcArgs<T> a, DevState *st) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = int(cl.block_rank()), nc = int(cl.num_blocks());
    extern __shared__ __align__(16) unsigned char lsm[];
    const int nv = a.nv, P = a.pitch, n = a.n;
    double *part = reinterpret_cast<double *>(lsm);       // kLzcWarps x nv
    double *recv = part + kLzcWarps * nv;                 // 2 x kLzcMaxCtas x nv
    double *tot = recv + 2 * kLzcMaxCtas * nv;            // nv
    double *la = tot + nv, *lb = la + kLzMax, *ls = lb + kLzMax, *sc = ls + kLzMax;  // sc: 8 scalars
    T *hT = reinterpret_cast<T *>(sc + 8);                // nv
    T *qs = hT + (nv + 1) / 2 * 2;                        // n
    T *ws = qs + (n + 1) / 2 * 2;                         // nr
    T *Qs = ws + (a.nr + 1) / 2 * 2;                      // nr x P
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row0 = rank * a.nr;
    const int nrows = max(0, min(a.nr, n - row0));
    int buf = 0;
    cl.sync();  // every CTA runs before another writes into its shared memory

    // tot[l] = sum over the cluster of part[warp][l], l < cnt (a fixed order)
    auto cluster_sum = [&](int cnt) {
        __syncthreads();
        const int l = tid >> 2, q = tid & 3;
        const bool in = l < cnt;
        double s = 0.0;
        if (warp * 8 < cnt) {  // warp-uniform
            if (in)
                for (int w = q; w < kLzcWarps; w += 4) s += part[w * nv + l];
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (in)
                for (int d = q; d < nc; d += 4)
                    *cl.map_shared_rank(recv + (buf * kLzcMaxCtas + rank) * nv + l, d) = s;
        }
        cl.sync();
        if (warp * 8 < cnt) {
            s = 0.0;
            if (in)
                for (int d = q; d < nc; d += 4) s += recv[(buf * kLzcMaxCtas + d) * nv + l];
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (in && q == 0) {
                tot[l] = s;
                hT[l] = T(s);
            }
        }
        buf ^= 1;
        __syncthreads();
    };
    // part[warp][slot] = the warp's sum of x (in x's type)
    auto warp_part = [&](auto x, int slot) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) part[warp * nv + slot] = double(x);
    };
    // ws[lr] (op) sum_l Qs[lr][l] hT[l], l < nvec; returns the thread's share of |ws|^2
    auto combine = [&](int nvec, bool subtract) -> T {
        T nrm = T(0);
        for (int b = 0; b < nrows; b += kLzcThreads / 4) {
            const int lr = b + (tid >> 2), q = tid & 3;
            T s = T(0);
            if (lr < nrows)
                for (int l = q; l < nvec; l += 4) s = fma(Qs[lr * P + l], hT[l], s);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (lr < nrows && q == 0) {
                const T x = subtract ? ws[lr] - s : s;
                ws[lr] = x;
                nrm = fma(x, x, nrm);
            }
        }
        return nrm;
    };
    // basis column j = ws * scale, sent to every CTA's qs; sc[4 + l] = s_l u_l^T q
    auto publish = [&](int j, T scale) {
        T *X = a.Q + int64_t(j & 1) * n;
        double u[kMaxLR] = {0.0, 0.0, 0.0, 0.0};
        for (int lr = tid; lr < nrows; lr += kLzcThreads) {
            const T q = ws[lr] * scale;
            Qs[lr * P + j] = q;
            X[row0 + lr] = q;
            for (int l = 0; l < v.lr_k; ++l) u[l] = fma(v.lr_u[int64_t(l) * n + row0 + lr], double(q), u[l]);
        }
        if (v.lr_k > 0) {
            for (int l = 0; l < v.lr_k; ++l) {
                const double x = warp_sum(u[l]);
                if (lane == 0) part[warp * nv + l] = x;
            }
            cluster_sum(v.lr_k);
            if (tid < v.lr_k) sc[4 + tid] = v.lr_s[tid] * tot[tid];
        } else {
            cl.sync();
        }
        for (int t = tid; t < n; t += kLzcThreads) qs[t] = __ldcg(X + t);
        __syncthreads();
    };
    // ws = S q on the CTA's rows, 8 lanes a row
    auto spmv = [&]() {
        for (int b = 0; b < nrows; b += kLzcThreads / 8) {
            const int lr = b + (tid >> 3), sub = tid & 7;
            T s = T(0);
            if (lr < nrows) {
                const int e1 = v.f_ptr[row0 + lr + 1];
                for (int e = v.f_ptr[row0 + lr] + sub; e < e1; e += 16) {
                    const bool two = e + 8 < e1;
                    const T c0 = v.f_val[e], c1 = two ? v.f_val[e + 8] : T(0);
                    const T x0 = qs[v.f_col[e]], x1 = two ? qs[v.f_col[e + 8]] : T(0);
                    s = fma(c0, x0, s);
                    if (two) s = fma(c1, x1, s);
                }
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lr < nrows && sub == 0) {
                s = fma(v.d_s[row0 + lr], qs[row0 + lr], s);
                for (int l = 0; l < v.lr_k; ++l) s = fma(T(v.lr_u[int64_t(l) * n + row0 + lr]), T(sc[4 + l]), s);
                ws[lr] = s;
            }
        }
        __syncthreads();
    };
    // tot[l] = q_l . w, l < nvec: lane l takes basis vector l, a warp its share of the rows
    auto project = [&](int nvec) {
        T s0 = T(0), s1 = T(0);
        for (int lr = warp; lr < nrows; lr += kLzcWarps) {
            const T w = ws[lr];
            if (lane < nvec) s0 = fma(Qs[lr * P + lane], w, s0);
            if (lane + 32 < nvec) s1 = fma(Qs[lr * P + lane + 32], w, s1);
        }
        if (lane < nvec) part[warp * nv + lane] = double(s0);
        if (lane + 32 < nvec) part[warp * nv + lane + 32] = double(s1);
        cluster_sum(nvec);
    };

    // start vector: seeded, or the previous Ritz vector plus a seeded one of norm 0.05
    {
        double nrm = 0.0;  // the norms of the start, the Ritz vector and the residual sum in FP64
        for (int lr = tid; lr < nrows; lr += kLzcThreads) {
            const uint64_t z = splitmix64_at(a.seed, uint64_t(row0 + lr));
            const T x = T(2.0 * (double(z >> 11) * (1.0 / 9007199254740992.0)) - 1.0);
            ws[lr] = x;
            nrm = fma(double(x), double(x), nrm);
        }
        warp_part(nrm, 0);
        cluster_sum(1);
        if (a.warm) {
            const T c = T(0.05 / sqrt(tot[0]));
            nrm = 0.0;
            for (int lr = tid; lr < nrows; lr += kLzcThreads) {
                const T x = a.Q[row0 + lr] + c * ws[lr];
                ws[lr] = x;
                nrm = fma(double(x), double(x), nrm);
            }
            warp_part(nrm, 0);
            cluster_sum(1);
        }
        if (tid == 0) sc[0] = tot[0] > 0.0 ? 1.0 / sqrt(tot[0]) : 0.0;
        __syncthreads();
        publish(0, T(sc[0]));
    }
    double theta = 0.0, resid = 0.0, anorm = 0.0;
    int m = 0, total = 0, stop = 0;
    for (int cycle = 0; cycle < a.max_restarts; ++cycle) {
        anorm = 0.0;
        stop = 0;
        for (int j = 0; j < a.kk; ++j) {
            spmv();
            project(j + 1);
            double alpha = tot[j];
            (void)combine(j + 1, true);
            __syncthreads();
            project(j + 1);
            alpha += tot[j];
            warp_part(combine(j + 1, true), 0);
            cluster_sum(1);
            if (tid == 0) {
                const double beta = sqrt(tot[0]);
                la[j] = alpha;
                lb[j] = beta;
                sc[1] = fmax(anorm, fabs(alpha) + beta + (j > 0 ? lb[j - 1] : 0.0));
                sc[0] = beta > 0.0 ? 1.0 / beta : 0.0;
                sc[2] = beta > 1e-13 * sc[1] ? 0.0 : 1.0;  // invariant subspace (or non-finite)
            }
            __syncthreads();
            anorm = sc[1];
            m = j + 1;
            stop = sc[2] != 0.0;
            if (stop) break;  // the same in every CTA: all hold the same sums
            if (j + 1 < a.kk) publish(j + 1, T(sc[0]));
        }
        total += m;
        __syncthreads();  // every thread has read sc
        if (warp == 0) {
            double rs = 0.0;
            const double th = warp_tridiag_min(la, lb, m, ls, &rs);
            if (lane == 0) {
                sc[1] = th;
                sc[2] = rs;
            }
            for (int l = lane; l < m; l += 32) hT[l] = T(ls[l]);
        }
        __syncthreads();
        theta = sc[1];
        resid = sc[2];
        warp_part(double(combine(m, false)), 0);
        cluster_sum(1);
        if (tid == 0) sc[0] = tot[0] > 0.0 ? 1.0 / sqrt(tot[0]) : 0.0;
        __syncthreads();
        publish(0, T(sc[0]));
        if (!isfinite(theta) || resid <= fmax(a.tol_rel * anorm, a.tol_abs) || stop) break;
    }
    // true residual of the final pair
    spmv();
    T r2 = T(0);
    for (int lr = tid; lr < nrows; lr += kLzcThreads) {
        const T d = ws[lr] - T(theta) * qs[row0 + lr];
        r2 = fma(d, d, r2);
    }
    warp_part(double(r2), 0);
    cluster_sum(1);
    if (rank == 0 && tid == 0) {
        st->theta = theta;
        st->resid_est = resid;
        st->anorm = anorm;
        st->lz_m = m;
        st->lz_total = total;
        st->lz_stop = stop;
        st->red[1] = tot[0];
    }
    cl.sync();  // no CTA leaves while another may still write into its shared memory
}

// ---------------------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------------------
// Whether the one-launch eigensolve takes vectors of v.n entries: its work runs on 16 of 152
// multiprocessors, so that long vectors are faster spread over all of them.  alm_lambda_min, ms,
// by launches / in one, ER graphs of degree 24 (the share of the SpMV grows with the degree: 400):
//   FP64   4000  2.61 / 2.00 (7.27 / 3.69)   6000  2.68 / 2.66 (7.37 / 5.17)   8192  6.52 / 8.18 (7.47 / 6.78)
//   FP32   4000  0.99 / 0.55 (2.59 / 1.04)   8192  2.78 / 1.94 (2.67 / 1.72)  12000  1.09 / 0.92 (8.01 / 6.92)
// At 8192 and degree 100 FP64 takes 5.62 / 6.45.  In FP32 one launch stays ahead up to where the basis
// no longer fits the cluster's shared memory (lzc_smem); its line is below that.
template <typename T>
static bool lz_cluster_rows(const SparseView<T> &v) {
    return v.n <= (sizeof(T) == 4 ? 8192 : 6000) || (v.n <= 8192 && v.nnz_u >= 125 * int64_t(v.n));
}
template <typename T>
static size_t lzc_smem(int n, int k, int ctas) {
    const int nv = k + 1 + kMaxLR, nr = (n + ctas - 1) / ctas, P = k | 1;
    const size_t dbl = size_t(kLzcWarps + 2 * kLzcMaxCtas + 1) * nv + 3 * kLzMax + 8;
    const size_t el = size_t((nv + 1) / 2 * 2) + (n + 1) / 2 * 2 + (nr + 1) / 2 * 2 + size_t(nr) * P;
    return 8 * dbl + sizeof(T) * el + 16;
}
template <typename T>
static cudaLaunchConfig_t lzc_config(const LaunchCtx &c, int ctas, size_t smem, cudaLaunchAttribute *at) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(ctas));
    cfg.blockDim = dim3(kLzcThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c.stream;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = unsigned(ctas);
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}
// CTAs of the cluster for the largest shared memory the kernel may ask for: 16 where the device
// schedules such a cluster, else 8, else none (0); asked once per precision
template <typename T>
static int lzc_ctas(const LaunchCtx &c, size_t *limit) {
    static std::mutex mu;
    static int ctas = -1;
    static size_t lim = 0;
    std::lock_guard<std::mutex> lk(mu);
    if (ctas < 0) {
        ctas = 0;
        int dev = 0, maxsm = 0;
        cudaFuncAttributes fa{};
        auto *fn = k_lz_cluster<T>;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaFuncGetAttributes(&fa, fn) == cudaSuccess &&
            cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess) {
            lim = size_t(maxsm) - fa.sharedSizeBytes;
            if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(lim)) == cudaSuccess &&
                cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
                for (int t = kLzcMaxCtas; t >= 8 && ctas == 0; t /= 2) {
                    cudaLaunchAttribute at{};
                    const cudaLaunchConfig_t cfg = lzc_config<T>(c, t, lim, &at);
                    int nclu = 0;
                    if (cudaOccupancyMaxActiveClusters(&nclu, fn, &cfg) == cudaSuccess && nclu > 0) ctas = t;
                }
        }
        (void)cudaGetLastError();
    }
    *limit = lim;
    return ctas;
}

template <typename T>
bool launch_lz_cluster(const LaunchCtx &c, const SparseView<T> &v, T *Q, int kk, int max_restarts, double tol_rel,
                       double tol_abs, uint64_t seed, bool warm) {
    if (!lz_cluster_rows(v)) return false;
    size_t limit = 0;
    const int ctas = lzc_ctas<T>(c, &limit);
    const size_t smem = ctas ? lzc_smem<T>(v.n, kk, ctas) : 0;
    if (ctas == 0 || smem > limit) return false;
    LzcArgs<T> a{Q, v.n, kk, kk | 1, (v.n + ctas - 1) / ctas, kk + 1 + kMaxLR, max_restarts, warm ? 1 : 0, tol_rel, tol_abs, seed};
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = lzc_config<T>(c, ctas, smem, &at);
    if (cudaLaunchKernelEx(&cfg, k_lz_cluster<T>, v, a, c.st) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    ++*c.launches;
    return true;
}

static inline int lz_grid(const LaunchCtx &c, int64_t n) {
    int64_t need = (n + kBlock - 1) / kBlock;
    if (need < 1) need = 1;
    return int(need < c.grid ? need : c.grid);
}

template <typename T>
void launch_lz_start(const LaunchCtx &c, T *q, int64_t n, uint64_t seed) {
    k_lz_start<T><<<lz_grid(c, n), kBlock, 0, c.stream>>>(q, n, seed, c.st, c.partials);
    ++*c.launches;
}

template <typename T>
void launch_lz_mix(const LaunchCtx &c, T *q, const T *u, int64_t n) {
    k_lz_mix<T><<<lz_grid(c, n), kBlock, 0, c.stream>>>(q, u, n, c.st, c.partials);
    ++*c.launches;
}

template <typename T>
void launch_lz_spmv(const LaunchCtx &c, const SparseView<T> &v, const T *q, T *w) {
    k_lz_spmv<T><<<lz_grid(c, v.n), kBlock, 0, c.stream>>>(v, q, w, c.st);
    ++*c.launches;
}

static inline int lz_tiles_grid(const LaunchCtx &c, int64_t n, int rpt) {
    const int64_t tiles = (n + int64_t(kBlock) * rpt - 1) / (int64_t(kBlock) * rpt);
    return int(tiles < c.grid ? tiles : c.grid);
}

// Four rows per thread amortise the per-tile warp sums; a vector too short to give every
// multiprocessor a tile that way takes one row per thread (more CTAs, shorter chains: the
// small eigensolves are latency-bound).
static inline bool lz_one_row(const LaunchCtx &c, int64_t n) {
    return (n + int64_t(kBlock) * 4 - 1) / (int64_t(kBlock) * 4) < int64_t(c.sms);
}

template <typename T>
void launch_lz_reorth(const LaunchCtx &c, const T *Q, int64_t ldq, int nvec, T *w, int64_t n, const double *h_in,
                      double *h_out, int j, int stage) {
    if (lz_one_row(c, n))
        k_lz_reorth<T, 1, false><<<lz_tiles_grid(c, n, 1), kBlock, 0, c.stream>>>(
            SparseView<T>{}, nullptr, nullptr, Q, ldq, nvec, w, n, h_in, h_out, j, stage, c.st, c.partials);
    else
        k_lz_reorth<T, 4, false><<<lz_tiles_grid(c, n, 4), kBlock, 0, c.stream>>>(
            SparseView<T>{}, nullptr, nullptr, Q, ldq, nvec, w, n, h_in, h_out, j, stage, c.st, c.partials);
    ++*c.launches;
}

template <typename T>
void launch_lz_spmv_reorth(const LaunchCtx &c, const SparseView<T> &v, const T *src, T *Q, int64_t ldq, T *w,
                           double *h_out, int j) {
    T *qj = Q + int64_t(j) * ldq;
    const int nvec = j + 1;
    if (lz_one_row(c, v.n))
        k_lz_reorth<T, 1, true><<<lz_tiles_grid(c, v.n, 1), kBlock, 0, c.stream>>>(
            v, src, qj, Q, ldq, nvec, w, v.n, nullptr, h_out, j, 0, c.st, c.partials);
    else
        k_lz_reorth<T, 4, true><<<lz_tiles_grid(c, v.n, 4), kBlock, 0, c.stream>>>(
            v, src, qj, Q, ldq, nvec, w, v.n, nullptr, h_out, j, 0, c.st, c.partials);
    ++*c.launches;
}

template <typename T>
void launch_lz_normalize(const LaunchCtx &c, const SparseView<T> &v, const T *src, T *dst, int64_t n, int mode,
                         int j) {
    k_lz_normalize<T><<<lz_grid(c, n), kBlock, 0, c.stream>>>(v, src, dst, n, mode, j, c.st, c.partials);
    ++*c.launches;
}

void launch_lz_tridiag(const LaunchCtx &c, int m) {
    k_lz_tridiag<<<1, 32, 0, c.stream>>>(c.st, m);
    ++*c.launches;
}

void launch_lz_reset(const LaunchCtx &c) {
    k_lz_reset<<<1, 32, 0, c.stream>>>(c.st);
    ++*c.launches;
}

template <typename T>
void launch_lz_ritz(const LaunchCtx &c, const T *Q, int64_t ldq, int m, T *dst, int64_t n) {
    k_lz_ritz<T><<<lz_grid(c, n), kBlock, 0, c.stream>>>(Q, ldq, m, dst, n, c.st, c.partials);
    ++*c.launches;
}

template <typename T>
void launch_lz_resid(const LaunchCtx &c, const T *w, const T *v, int64_t n) {
    k_lz_resid<T><<<lz_grid(c, n), kBlock, 0, c.stream>>>(w, v, n, c.st, c.partials);
    ++*c.launches;
}

#define ALM_LZ_INST(T)                                                                                          \
    template bool launch_lz_cluster<T>(const LaunchCtx &, const SparseView<T> &, T *, int, int, double, double, \
                                       uint64_t, bool);                                                         \
    template void launch_lz_start<T>(const LaunchCtx &, T *, int64_t, uint64_t);                                \
    template void launch_lz_mix<T>(const LaunchCtx &, T *, const T *, int64_t);                                 \
    template void launch_lz_spmv<T>(const LaunchCtx &, const SparseView<T> &, const T *, T *);                  \
    template void launch_lz_reorth<T>(const LaunchCtx &, const T *, int64_t, int, T *, int64_t, const double *, \
                                      double *, int, int);                                                      \
    template void launch_lz_spmv_reorth<T>(const LaunchCtx &, const SparseView<T> &, const T *, T *, int64_t, T *, \
                                           double *, int);                                                      \
    template void launch_lz_normalize<T>(const LaunchCtx &, const SparseView<T> &, const T *, T *, int64_t, int, \
                                         int);                                                                  \
    template void launch_lz_ritz<T>(const LaunchCtx &, const T *, int64_t, int, T *, int64_t);                  \
    template void launch_lz_resid<T>(const LaunchCtx &, const T *, const T *, int64_t);

ALM_LZ_INST(float)
ALM_LZ_INST(double)

}  // namespace alm
