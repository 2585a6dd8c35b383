// Float-pair ("double-float") helpers of the FP32 form: a double split into two floats,
// compensated accumulation of a lane's 4-vector of sum_k s_k x_k, and the compensated
// squared norm of an R row over its row group.  Shared by the per-kernel path and the
// batched persistent solver.
#pragma once

#include "dev_util.cuh"

namespace alm {

__device__ __forceinline__ void split_pair(double d, float &hi, float &lo) {
    hi = float(d);
    lo = float(d - double(hi));
}
__device__ __forceinline__ void split_pair(double d, double &hi, double &lo) {
    hi = d;
    lo = 0.0;
}
// Accumulator of a lane's vector of sum_k s_k x_k: plain FMAs in the FP64 form,
// compensated (products split exactly with FMA, sums with two-sum) in the FP32 form so
// that G = 2 S R keeps its accuracy when its O(|S||R|) terms cancel.
struct AccD {
    double2 v;
    __device__ __forceinline__ void init() { v = make_double2(0.0, 0.0); }
    __device__ __forceinline__ void add(double s, double2 x) { v = fma4(s, x, v); }
    __device__ __forceinline__ void add_lo(double s, double2 x) { v = fma4(s, x, v); }
    __device__ __forceinline__ double2 value() const { return v; }
    // add up the accumulators of lanes FROM, 2 FROM, .. < TO apart
    template <int FROM, int TO>
    __device__ __forceinline__ void merge(unsigned mask) {
#pragma unroll
        for (int o = FROM; o < TO; o <<= 1) {
            v.x += __shfl_xor_sync(mask, v.x, o);
            v.y += __shfl_xor_sync(mask, v.y, o);
        }
    }
    static constexpr int kWords = 1;  // W-vectors of its state
    __device__ __forceinline__ void store(double *p) const { stv(p, v); }
    __device__ __forceinline__ void add_stored(const double *p) { v = fma4(1.0, ld(p), v); }
};
struct AccF {
    float hi[4], lo[4];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int k = 0; k < 4; ++k) hi[k] = lo[k] = 0.f;
    }
    __device__ __forceinline__ void add(float s, float4 x) {
        const float c[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float p = s * c[k];
            lo[k] += fmaf(s, c[k], -p);
            two_sum_acc(hi[k], lo[k], p);
        }
    }
    __device__ __forceinline__ void add_lo(float s, float4 x) {  // small correction terms
        lo[0] = fmaf(s, x.x, lo[0]);
        lo[1] = fmaf(s, x.y, lo[1]);
        lo[2] = fmaf(s, x.z, lo[2]);
        lo[3] = fmaf(s, x.w, lo[3]);
    }
    template <int FROM, int TO>
    __device__ __forceinline__ void merge(unsigned mask) {
#pragma unroll
        for (int o = FROM; o < TO; o <<= 1)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float h2 = __shfl_xor_sync(mask, hi[k], o), l2 = __shfl_xor_sync(mask, lo[k], o);
                two_sum_acc(hi[k], lo[k], h2);
                lo[k] += l2;
            }
    }
    static constexpr int kWords = 2;
    __device__ __forceinline__ void store(float *p) const {
        stv(p, make_float4(hi[0], hi[1], hi[2], hi[3]));
        stv(p + 4, make_float4(lo[0], lo[1], lo[2], lo[3]));
    }
    __device__ __forceinline__ void add_stored(const float *p) {
        const float4 h = ld(p), l = ld(p + 4);
        two_sum_acc(hi[0], lo[0], h.x);
        two_sum_acc(hi[1], lo[1], h.y);
        two_sum_acc(hi[2], lo[2], h.z);
        two_sum_acc(hi[3], lo[3], h.w);
        lo[0] += l.x;
        lo[1] += l.y;
        lo[2] += l.z;
        lo[3] += l.w;
    }
    __device__ __forceinline__ float4 value() const {
        return make_float4(hi[0] + lo[0], hi[1] + lo[1], hi[2] + lo[2], hi[3] + lo[3]);
    }
};
template <typename T>
struct AccOf;
template <>
struct AccOf<float> {
    using type = AccF;
};
template <>
struct AccOf<double> {
    using type = AccD;
};

// Error-free accumulation against a power-of-two bias (the extraction step of Rump, Ogita and
// Oishi, "Accurate floating-point summation", SIAM J. Sci. Comput. 31, 2008).  `sg` starts at
// bias = 1.5 * 2^e with 2^e above twice every partial sum, so sg stays in (2^e, 2^(e+1)).  One
// FMA rounds the exact sum sg + c x; q = s - sg is then exact (Sterbenz: s and sg lie within a
// factor of two) and c x - q, the part of c x that the rounding dropped, is exact when c x is
// a float (c a power of two) and otherwise off by 2^-24 of a unit in the last place of sg:
// it goes to `lo`.  Four operations per term, the product included, against eight to ten for a
// product error plus a two-sum.  If a bound is exceeded the sum loses only the exactness of
// that step (plain FP32 rounding).
__device__ __forceinline__ void ext_fma(float &sg, float &lo, float c, float x) {
    const float s = fmaf(c, x, sg);
    const float q = s - sg;
    lo += fmaf(c, x, -q);
    sg = s;
}
// 1.5 * 2^e with 2^e the power of two just above 2 b (b >= 0), capped below the overflow range
__device__ __forceinline__ float ext_bias(float b) {
    unsigned u = __float_as_uint(2.f * b) & 0x7f800000u;
    u = u < 0x7e000000u ? u : 0x7e000000u;
    return __uint_as_float(u + 0x00c00000u);
}
// c x accumulated into (sg, lo) per component
__device__ __forceinline__ void ext_term(float (&sg)[4], float (&lo)[4], float c, float4 x) {
    ext_fma(sg[0], lo[0], c, x.x);
    ext_fma(sg[1], lo[1], c, x.y);
    ext_fma(sg[2], lo[2], c, x.z);
    ext_fma(sg[3], lo[3], c, x.w);
}

// The lane's a . b as a float pair (products split exactly, sums with two-sum): the constraint
// values, whose residual is far smaller than they are and is multiplied by sigma.  The FP64
// form returns its plain sum in hi.
__device__ __forceinline__ void dot_pair(float4 a, float4 b, float &hi, float &lo) {
    const float x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
    hi = x[0] * y[0];
    lo = fmaf(x[0], y[0], -hi);
#pragma unroll
    for (int k = 1; k < 4; ++k) {
        const float p = x[k] * y[k];
        lo += fmaf(x[k], y[k], -p);
        two_sum_acc(hi, lo, p);
    }
}
__device__ __forceinline__ void dot_pair(double2 a, double2 b, double &hi, double &lo) {
    hi = dot(a, b);
    lo = 0.0;
}
// sum of the pairs over the LANES lanes of a row
template <int LANES>
__device__ __forceinline__ void pair_group_sum(float &hi, float &lo, unsigned mask) {
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(mask, hi, o), l2 = __shfl_xor_sync(mask, lo, o);
        two_sum_acc(hi, lo, h2);
        lo += l2;
    }
}
template <int LANES>
__device__ __forceinline__ void pair_group_sum(double &hi, double &, unsigned mask) {
    hi = group_sum<LANES>(hi, mask);
}

// float-pair sum of squares of a lane's vector over the row group (FP32 form); the
// FP64 form returns its plain sum in hi
__device__ __forceinline__ void norm2_pair(float4 v, unsigned mask, int lanes, float &hi, float &lo) {
    const float c[4] = {v.x, v.y, v.z, v.w};
    hi = c[0] * c[0];  // the pair starts from the first square (a two-sum into 0 is exact)
    lo = fmaf(c[0], c[0], -hi);
#pragma unroll
    for (int k = 1; k < 4; ++k) {
        const float p = c[k] * c[k];
        lo += fmaf(c[k], c[k], -p);
        two_sum_acc(hi, lo, p);
    }
    for (int o = lanes / 2; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(mask, hi, o);
        const float l2 = __shfl_xor_sync(mask, lo, o);
        two_sum_acc(hi, lo, h2);
        lo += l2;
    }
}
__device__ __forceinline__ void norm2_pair(double2 v, unsigned mask, int lanes, double &hi, double &lo) {
    double x = v.x * v.x + v.y * v.y;
    for (int o = lanes / 2; o > 0; o >>= 1) x += __shfl_xor_sync(mask, x, o);
    hi = x;
    lo = 0.0;
}

}  // namespace alm
