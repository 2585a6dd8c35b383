// Exact minimiser of the line-search quartic phi(a) = q0 + q1 a + ... + q4 a^4 over
// a >= 0 (the closed-form step of the inner loop), in FP64.  Shared by the per-kernel
// inner loop and the batched persistent solver.
#pragma once

#include <cmath>

namespace alm {

// ---------------------------------------------------------------------------------------
// exact minimiser of the quartic phi(a) = q0 + q1 a + q2 a^2 + q3 a^3 + q4 a^4 on a >= 0
// ---------------------------------------------------------------------------------------
__device__ inline int real_cubic_roots64(double c3, double c2, double c1, double c0, double x[3]) {
    // The same in FP64 throughout, where the FP32 start is too coarse.  Depressed cubic t^3 + p t + q = 0 with
    // x = t - B/3 (Cardano; trigonometric form when all three roots are real).
    const double B = c2 / c3, Cc = c1 / c3, Dd = c0 / c3;
    const double p = Cc - B * B / 3.0;
    const double q = 2.0 * B * B * B / 27.0 - B * Cc / 3.0 + Dd;
    const double shift = -B / 3.0;
    const double disc = q * q / 4.0 + p * p * p / 27.0;
    int nr;
    if (disc > 0.0) {
        const double sd = sqrt(disc);
        x[0] = cbrt(-q / 2.0 + sd) + cbrt(-q / 2.0 - sd) + shift;
        nr = 1;
    } else if (p == 0.0) {
        x[0] = shift;
        nr = 1;
    } else {
        const double rr = 2.0 * sqrt(-p / 3.0);
        double arg = (3.0 * q / (2.0 * p)) * sqrt(-3.0 / p);
        arg = fmin(1.0, fmax(-1.0, arg));
        const double ph = acos(arg) / 3.0;
        const double tpi3 = 2.0943951023931954923;  // 2 pi / 3
        for (int k = 0; k < 3; ++k) x[k] = rr * cos(ph - tpi3 * k) + shift;
        nr = 3;
    }
    for (int k = 0; k < nr; ++k) {  // Newton polish on the original cubic
        double t = x[k];
        for (int it = 0; it < 4; ++it) {
            const double f = ((c3 * t + c2) * t + c1) * t + c0;
            const double fp = (3.0 * c3 * t + 2.0 * c2) * t + c1;
            if (fp == 0.0) break;
            const double nt = t - f / fp;
            if (!isfinite(nt)) break;
            t = nt;
        }
        x[k] = t;
    }
    // The discriminant's sign is its rounding's when two roots lie some 1e8 times below the third: the
    // quadratic that the largest root leaves over (divided out from the low end, which is the stable
    // way for it) tells whether there are two more.
    double xm = x[0];
    for (int k = 1; k < nr; ++k)
        if (fabs(x[k]) > fabs(xm)) xm = x[k];
    const double g = -c0 / xm, b = (g - c1) / xm;  // (x - xm)(c3 x^2 + b x + g)
    const double d2 = b * b - 4.0 * c3 * g;
    if (!(d2 > 0.0) || !isfinite(d2)) return nr;
    const double h = -0.5 * (b + copysign(sqrt(d2), b));
    const double two[2] = {h / c3, g / h};
    for (int k = 0; k < 2; ++k) {
        double t = two[k];
        for (int it = 0; it < 4; ++it) {
            const double f = ((c3 * t + c2) * t + c1) * t + c0;
            const double fp = (3.0 * c3 * t + 2.0 * c2) * t + c1;
            const double nt = t - f / fp;
            if (!isfinite(nt)) break;
            t = nt;
        }
        x[k + 1] = t;
    }
    x[0] = xm;
    return 3;
}

// FP64 on this part: 64 cycles an instruction for the one thread that runs this, 568 a division,
// more for cbrt, acos and cos; the step waits for it.  So the roots are located in FP32 on the
// cubic scaled to coefficients of about 1 and polished by Newton in FP64, with reciprocals by the
// hardware's approximation and two Newton steps.  Cycles for the minimiser, FP64 cbrt, acos, cos
// and divisions throughout -> so: one root 21,000 -> 7,000, three roots 33,000 -> 12,000.
__device__ __forceinline__ double quick_rcp(double d) {
    const double m = fabs(d);
    if (!(m > 1e-290 && m < 1e290)) return 1.0 / d;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    r = fma(r, fma(-d, r, 1.0), r);
    return fma(r, fma(-d, r, 1.0), r);
}
// floor(log2 |x|) of a normal x, a large negative number for 0
__device__ __forceinline__ int exponent_of(double x) {
    const int e = (__double2hiint(x) >> 20) & 0x7ff;
    return e ? e - 1023 : -4096;
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// real roots of c3 x^3 + c2 x^2 + c1 x + c0, c3 != 0
__device__ inline int real_cubic_roots(double c3, double c2, double c1, double c0, double x[3]) {
    const double ic = quick_rcp(c3);
    double B = c2 * ic, Cc = c1 * ic, Dd = c0 * ic;  // monic
    if (!isfinite(B) || !isfinite(Cc) || !isfinite(Dd)) return 0;
    int e = exponent_of(B);  // x = 2^e t: the largest coefficient of t's cubic is about 1
    e = max(e, (exponent_of(Cc) + 1) >> 1);
    e = max(e, (exponent_of(Dd) + 2) / 3);
    e = e < -300 ? 0 : min(e, 300);
    const double s = pow2(-e);
    B *= s;
    Cc *= s * s;
    Dd *= s * s * s;
    // depressed cubic u^3 + p u + q = 0 with t = u - B/3 (Cardano; trigonometric form when all
    // three roots are real)
    const double b3 = B * (1.0 / 3.0);
    const double p = fma(-B, b3, Cc);
    const double q = fma(b3, fma(2.0 * b3, b3, -Cc), Dd);
    const double hq = 0.5 * q, p3 = p * (1.0 / 3.0);
    const double disc = fma(hq, hq, p3 * p3 * p3);
    const float pf = float(p3), qf = float(hq), shift = float(-b3);
    float t0[3];
    int nr = 1;
    if (disc > 0.0) {
        const float sd = sqrtf(float(disc));
        const float u = cbrtf(qf > 0.f ? -qf - sd : -qf + sd);  // no cancellation
        t0[0] = (u != 0.f ? u - pf / u : 0.f) + shift;
    } else if (!(pf < 0.f)) {
        t0[0] = shift;
    } else {
        const float rr = sqrtf(-pf);
        const float ph = acosf(fminf(1.f, fmaxf(-1.f, -qf / (rr * rr * rr)))) * (1.f / 3.f);
        for (int k = 0; k < 3; ++k) t0[k] = 2.f * rr * cosf(ph - 2.0943951f * float(k)) + shift;
        nr = 3;
    }
    // The FP32 starts do for roots of similar size.  Where roots lie far below the largest (a cubic
    // whose leading coefficient is small: -0.17 + 4.8e-6 a + 4.5 a^3 + 2e-8 a^4 has its minimum at 0.11
    // and a stationary point at -1.7e8) they may not: a discriminant within rounding of its terms does not
    // tell one real root from three, and two starts can end on one root.  Both are seen here, as is a
    // Newton that has not converged, and FP64 throughout takes over.
    bool ok = nr == 3 || disc > 0x1p-20 * fma(hq, hq, fabs(p3 * p3 * p3));
    double t1[3];
    for (int k = 0; k < nr; ++k) {  // Newton on the scaled cubic
        double t = double(t0[k]);
        bool conv = false;
        for (int it = 0; it < 6 && !conv; ++it) {
            const double f = fma(fma(t + B, t, Cc), t, Dd);
            const double fp = fma(fma(3.0, t, 2.0 * B), t, Cc);
            if (fp == 0.0) break;
            const double d = f * quick_rcp(fp);
            if (!isfinite(d)) break;
            t -= d;
            conv = fabs(d) <= 0x1p-30 * fabs(t);  // the error is now its square
        }
        ok = ok && conv;
        t1[k] = t;
        x[k] = t * pow2(e);
        for (int l = 0; l < k; ++l) ok = ok && fabs(t - t1[l]) > 0x1p-16 * fmax(fabs(t), fabs(t1[l]));
    }
    if (!ok) return real_cubic_roots64(c3, c2, c1, c0, x);
    return nr;
}

__device__ __forceinline__ double quartic_drop(const double q[5], double a) {  // phi(a) - phi(0)
    return a * (q[1] + a * (q[2] + a * (q[3] + a * q[4])));
}

__device__ inline double quartic_argmin(const double q[5], int *unbounded) {
    *unbounded = 0;
    if (q[4] < 0.0 || (q[4] == 0.0 && (q[3] < 0.0 || (q[3] == 0.0 && (q[2] < 0.0 || (q[2] == 0.0 && q[1] < 0.0)))))) {
        *unbounded = 1;
        return INFINITY;
    }
    double cand[3];
    int nc = 0;
    if (q[4] > 0.0) {
        nc = real_cubic_roots(4.0 * q[4], 3.0 * q[3], 2.0 * q[2], q[1], cand);
    } else if (q[3] > 0.0) {  // phi' = 3 q3 a^2 + 2 q2 a + q1
        const double A = 3.0 * q[3], Bq = 2.0 * q[2], Cq = q[1];
        const double disc = Bq * Bq - 4.0 * A * Cq;
        if (disc >= 0.0) {
            const double sd = sqrt(disc);
            cand[0] = (-Bq - sd) / (2.0 * A);
            cand[1] = (-Bq + sd) / (2.0 * A);
            nc = 2;
        }
    } else if (q[2] > 0.0) {
        cand[0] = -q[1] / (2.0 * q[2]);
        nc = 1;
    }
    for (int a = 0; a < nc; ++a)  // ascending: the smallest of equal minima wins
        for (int b = a + 1; b < nc; ++b)
            if (cand[b] < cand[a]) { const double t = cand[a]; cand[a] = cand[b]; cand[b] = t; }
    double best = 0.0, bestv = 0.0;
    for (int k = 0; k < nc; ++k) {
        const double a = cand[k];
        if (!(a > 0.0) || !isfinite(a)) continue;
        const double v = quartic_drop(q, a);
        if (v < bestv) { best = a; bestv = v; }
    }
    return best;
}

}  // namespace alm
