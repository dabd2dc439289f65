// Per-thread accumulation of scalar products, accurate to FP64 and beyond.
//
// FP64: one FMA per term.  FP32: a product of two FP32 values is exact in FP64, but
// forming it there takes two conversions and an FMA on a pipe of 1.7 lanes per
// clock and SM.  Here it is split into an FP32 pair (product and FMA remainder),
// and the pairs are added into three FP32 numbers by two-sums, so that a
// thread's sum keeps about 70 bits; FP64 begins with get().  Packed arithmetic,
// two terms per lane and instruction.  The split needs products inside the
// range of FP32: ok() is false where a term overflowed, is not finite, or
// the largest is so small that the remainders may have underflowed (zero among
// them), and the caller then sums its terms on another scale or in FP64.
#pragma once
#include <cuda_runtime.h>

namespace wvl {

template <typename T> struct DotAcc;

template <> struct DotAcc<double> {
    double v = 0.0;
    __device__ __forceinline__ void add(double x, double y) { v = fma(x, y, v); }
    __device__ __forceinline__ double get() const { return v; }
    __device__ __forceinline__ bool ok() const { return true; }
};

template <> struct DotAcc<float> {
    float2 s{0.f, 0.f}, c{0.f, 0.f}, d{0.f, 0.f};
    float pmax = 0.f;
    // a += x exactly: returns what the sum lost
    __device__ __forceinline__ static float2 two_sum(float2& a, float2 x) {
        const float2 m1 = make_float2(-1.f, -1.f);
        const float2 t = __fadd2_rn(a, x);
        const float2 b = __ffma2_rn(a, m1, t);       // t - a
        const float2 r = __ffma2_rn(b, m1, t);       // t - b
        const float2 e1 = __ffma2_rn(r, m1, a);      // a - (t - b)
        const float2 e2 = __ffma2_rn(b, m1, x);      // x - b
        a = t;
        return __fadd2_rn(e1, e2);
    }
    __device__ __forceinline__ void add(float2 x, float2 y) {
        const float2 p = __fmul2_rn(x, y);
        const float2 e = __ffma2_rn(x, y, make_float2(-p.x, -p.y));
        const float2 r = two_sum(s, p);
        const float2 r1 = two_sum(c, r);
        const float2 r2 = two_sum(c, e);
        d = __fadd2_rn(d, __fadd2_rn(r1, r2));
        pmax = fmaxf(pmax, fmaxf(fabsf(p.x), fabsf(p.y)));
    }
    __device__ __forceinline__ void add(float x, float y) { add(make_float2(x, 0.f), make_float2(y, 0.f)); }
    __device__ __forceinline__ double get() const {
        const double lo = ((double)d.x + (double)d.y) + ((double)c.x + (double)c.y);
        return ((double)s.x + (double)s.y) + lo;
    }
    // largest product in [2^-60, 2^100]; the sums finite (a NaN or an infinity shows in s)
    __device__ __forceinline__ bool ok() const {
        return (pmax >= 8.7e-19f && pmax <= 1.2e30f) && fabsf(s.x) < 1e35f && fabsf(s.y) < 1e35f;
    }
};

}  // namespace wvl
