// Smallest eigenpair of a symmetric tridiagonal matrix in FP64 (the Lanczos matrix T of a
// restart cycle), computed by one warp.  Shared by the per-kernel Lanczos and the batched
// persistent solver.
//
// Bound: one warp issues an FP64 instruction every 64 cycles on this part (measured, whatever
// the number of active lanes) and a division costs 568, so the time is the length of the FP64
// chain.  Hence: the bracket comes from a multisection in FP32 (32 points a round, no FP64);
// FP64 does inverse iteration with shifts below the eigenvalue, where T - sigma I is positive
// definite and needs no pivoting, and each factorisation burns from both ends to the middle
// row, lane 0 from the top and lane 1 from the bottom, which halves its chain.  The shift
// follows the Rayleigh quotient theta: sigma = theta - |T x - theta x| is below the eigenvalue
// next to theta, and a factorisation that meets a pivot <= 0 shows that a smaller eigenvalue
// exists, whereupon the shift moves down.  The last factorisation succeeds at a shift within
// rounding of theta: it proves that theta is the smallest eigenvalue, as a Sturm count does.
// A 32 x 32 matrix: 324 us with an FP64 Sturm multisection and three pivoted factorisations,
// 145 us with minors in place of pivots, 50 us this way (eigenvalue and residual within 5e-16 of
// the norm over random, clustered, graded and split matrices of 1 to 64 rows).
#pragma once

#include <cfloat>
#include <cmath>

#include "alm_internal.h"

namespace alm {

struct TridiagScratch {
    double a[kLzMax], b[kLzMax];   // T scaled to entries of at most 1
    double l[kLzMax], rd[kLzMax];  // b / pivot towards the middle row, 1 / pivot
    double x[kLzMax], y[kLzMax];
    float af[kLzMax], b2f[kLzMax];
};

__device__ __forceinline__ double tri_warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// 1 / d for normal d > 0: the hardware's approximation and two Newton steps (20 -> 40 -> full
// bits; 276 cycles in place of the correctly rounded division's 568)
__device__ __forceinline__ double tri_rcp(double d) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    r = fma(r, fma(-d, r, 1.0), r);
    return fma(r, fma(-d, r, 1.0), r);
}

// Factor T - sigma I from both ends to row mid = m / 2; whether every pivot is positive.
__device__ __forceinline__ bool tri_factor(TridiagScratch &s, int m, double sigma) {
    const int lane = threadIdx.x & 31, mid = m / 2;
    bool ok = true;
    if (lane < 2) {
        const int dir = lane == 0 ? 1 : -1;
        const int n = lane == 0 ? mid : m - 1 - mid;  // rows of this end
        int i = lane == 0 ? 0 : m - 1;
        double bl = 0.0;  // b l of the row before
        for (int t = 0; t < n; ++t, i += dir) {
            const double d = (s.a[i] - sigma) - bl;
            ok = ok && d > 0.0;
            const double r = tri_rcp(d), b = s.b[lane == 0 ? i : i - 1];
            const double l = b * r;
            s.rd[i] = r;
            s.l[i] = l;
            bl = b * l;
        }
        const double bl1 = __shfl_sync(0x3u, bl, 1);
        if (lane == 0) {
            const double d = ((s.a[mid] - sigma) - bl) - bl1;
            ok = ok && d > 0.0;
            s.rd[mid] = tri_rcp(d);
        }
    }
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();
    return ok;
}

// x <- (T - sigma I)^{-1} x with the factors of tri_factor; normalise: then |x| = 1
__device__ __forceinline__ void tri_solve(TridiagScratch &s, int m, bool normalise) {
    const int lane = threadIdx.x & 31, mid = m / 2;
    if (lane < 2) {
        const int dir = lane == 0 ? 1 : -1;
        const int n = lane == 0 ? mid : m - 1 - mid;
        int i = lane == 0 ? 0 : m - 1;
        double ly = 0.0;
        for (int t = 0; t < n; ++t, i += dir) {
            const double y = s.x[i] - ly;
            s.y[i] = y;
            ly = s.l[i] * y;
        }
        const double ly1 = __shfl_sync(0x3u, ly, 1);
        double x = 0.0;
        if (lane == 0) {
            x = ((s.x[mid] - ly) - ly1) * s.rd[mid];
            s.x[mid] = x;
        }
        x = __shfl_sync(0x3u, x, 0);
        for (int t = 0; t < n; ++t) {
            i -= dir;
            x = fma(-s.l[i], x, s.y[i] * s.rd[i]);
            s.x[i] = x;
        }
    }
    __syncwarp();
    if (!normalise) return;
    double nx = 0.0;
    for (int i = lane; i < m; i += 32) nx = fma(s.x[i], s.x[i], nx);
    nx = tri_warp_sum(nx);
    const bool good = nx > 0.0 && isfinite(nx);
    const double inx = good ? rsqrt(nx) : 0.0;
    for (int i = lane; i < m; i += 32) s.x[i] = good ? s.x[i] * inx : double(i == 0);
    __syncwarp();
}

// theta = x^T T x; returns |T x - theta x|
__device__ __forceinline__ double tri_rayleigh(const TridiagScratch &s, int m, double &theta) {
    const int lane = threadIdx.x & 31;
    double t[(kLzMax + 31) / 32], q = 0.0;
#pragma unroll
    for (int k = 0; k < (kLzMax + 31) / 32; ++k) {
        const int i = lane + 32 * k;
        t[k] = 0.0;
        if (i >= m) continue;
        t[k] = s.a[i] * s.x[i];
        if (i > 0) t[k] = fma(s.b[i - 1], s.x[i - 1], t[k]);
        if (i + 1 < m) t[k] = fma(s.b[i], s.x[i + 1], t[k]);
        q = fma(s.x[i], t[k], q);
    }
    theta = tri_warp_sum(q);
    double r2 = 0.0;
#pragma unroll
    for (int k = 0; k < (kLzMax + 31) / 32; ++k) {
        const int i = lane + 32 * k;
        if (i >= m) continue;
        const double r = fma(-theta, s.x[i], t[k]);
        r2 = fma(r, r, r2);
    }
    return sqrt(tri_warp_sum(r2));
}

// a[0..m-1] (diagonal) and b[0..m-2] (off-diagonal; b[m-1] = the next Lanczos beta, used
// for the residual estimate) are read by every lane; 1 <= m <= kLzMax.  Every lane of the
// calling warp must call it, and one warp of the block only.  Writes the unit eigenvector to
// x_out[0..m-1] (visible to the warp on return) and, lane 0, the residual estimate
// |b[m-1] x[m-1]| to *resid_out; the eigenvalue is returned to all lanes (NaN for a matrix
// with a non-finite entry).
__device__ inline double warp_tridiag_min(const double *a, const double *b, int m, double *x_out,
                                          double *resid_out) {
    __shared__ TridiagScratch s;
    const int lane = threadIdx.x & 31;
    // scale to entries of at most 1 by a power of two (exact)
    bool fin = true;
    for (int i = lane; i < m; i += 32) {
        const double bi = i + 1 < m ? b[i] : 0.0;
        fin = fin && isfinite(a[i]) && isfinite(bi);
        s.a[i] = fabs(a[i]);
        s.b[i] = fabs(bi);
    }
    __syncwarp();
    if (!__all_sync(0xffffffffu, fin)) {
        for (int i = lane; i < m; i += 32) x_out[i] = double(i == 0);
        if (lane == 0) *resid_out = NAN;
        __syncwarp();
        return NAN;
    }
    int ex = -2000;  // exponent of the largest entry
    for (int i = lane; i < m; i += 32) {
        if (s.a[i] > 0.0) ex = max(ex, ilogb(s.a[i]) + 1);
        if (s.b[i] > 0.0) ex = max(ex, ilogb(s.b[i]) + 1);
    }
    ex = __reduce_max_sync(0xffffffffu, ex);
    if (ex == -2000) ex = 0;
    __syncwarp();
    for (int i = lane; i < m; i += 32) {
        s.a[i] = ldexp(a[i], -ex);
        s.b[i] = i + 1 < m ? ldexp(b[i], -ex) : 0.0;
        s.af[i] = float(s.a[i]);
        const float bf = float(s.b[i]);
        s.b2f[i] = bf * bf;
        s.x[i] = 1.0 + 0.5 * double(sinf(float(i) + 1.f));
    }
    __syncwarp();
    // FP32 multisection on the pivots' signs from the Gershgorin bracket (within [-3, 3])
    float lo = 4.f, hi = -4.f;
    for (int i = lane; i < m; i += 32) {
        const float rad = (i > 0 ? fabsf(float(s.b[i - 1])) : 0.f) + fabsf(float(s.b[i]));
        lo = fminf(lo, s.af[i] - rad);
        hi = fmaxf(hi, s.af[i] + rad);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const float low = lo - 1e-5f;  // below every eigenvalue
    for (int round = 0; round < 8 && hi - lo > 1e-6f; ++round) {
        const float step = (hi - lo) * (1.f / 33.f);
        const float x = lo + step * float(lane + 1);
        float d = s.af[0] - x;
        bool pos = d > 0.f;
        for (int i = 1; i < m; ++i) {
            d = (s.af[i] - x) - __fdividef(s.b2f[i - 1], d);
            pos = pos && d > 0.f;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, !pos);
        const int f = bal ? __ffs(bal) - 1 : 32;
        const float nhi = f < 32 ? lo + step * float(f + 1) : hi;
        lo = f > 0 ? lo + step * float(f) : lo;
        hi = nhi;
    }
    // inverse iteration below the eigenvalue; sigma_ok: the largest shift shown to be below it
    const double delta = 16.0 * DBL_EPSILON;
    double sigma = double(lo) - 1e-5, sigma_ok = double(low), theta = 0.0, width = 1.0;
    for (int it = 0; it < 64; ++it) {
        if (tri_factor(s, m, sigma)) {
            if (width <= delta) {
                tri_solve(s, m, true);
                break;
            }
            tri_solve(s, m, false);
            tri_solve(s, m, true);
            sigma_ok = sigma;
            width = fmax(delta, tri_rayleigh(s, m, theta));
            sigma = fmax(theta - width, sigma_ok);
        } else {  // an eigenvalue lies below sigma
            width = 1.0;
            sigma = sigma_ok + 0.5 * (sigma - sigma_ok);
            if (!(sigma > sigma_ok + 0.5 * DBL_EPSILON)) {
                sigma = sigma_ok - delta;
                width = delta;
            }
        }
    }
    (void)tri_rayleigh(s, m, theta);
    for (int i = lane; i < m; i += 32) x_out[i] = s.x[i];
    if (lane == 0) *resid_out = fabs(b[m - 1] * s.x[m - 1]);
    __syncwarp();
    return ldexp(theta, ex);
}

}  // namespace alm
