// Shared by the fused chain's kernels (fused_kernel.cu, fused_plane.cu).
#pragma once
#include <cuda_runtime.h>

#include "pass_kernel.cuh"
#include "static_for.cuh"

namespace wvl {
namespace {

// Energy accumulator of an energy partial (one CTA's share of Ekin): FP64
// in the FP64 form; in the FP32 form a compensated FP32 pair (two-sum,
// about 48 bits) of the item chains of at most 32 products, carried through
// the warp's shuffle tree and formed in FP64 from the warp on, as the
// potential kernel does for Epot -- FP64 additions through the tree took
// about 12 % of the last column kernel on GB300's narrow FP64 pipe.
template <typename T> struct EAcc;
template <> struct EAcc<double> {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ double warp_sum() {
        double t = v;
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        return t;
    }
};
template <> struct EAcc<float> {
    FF f{0.f, 0.f};
    __device__ __forceinline__ void add(float x) { ff_add(f, x); }
    __device__ __forceinline__ double warp_sum() {
        FF g = f;
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_down_sync(0xffffffffu, g.hi, o);
            const float ol = __shfl_down_sync(0xffffffffu, g.lo, o);
            ff_add(g, oh);
            g.lo += ol;
        }
        return (double)g.hi + (double)g.lo;
    }
};
// the CTA's sum: the warps' sums, then warp 0 adds them in a fixed tree
template <typename T>
__device__ __forceinline__ double fz_block_sum(EAcc<T>& e, double* red) {
    const double w = e.warp_sum();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (int)(blockDim.x >> 5);
    if (lane == 0) red[warp] = w;
    __syncthreads();
    double t = 0.0;
    if (warp == 0) {
        t = lane < nw ? red[lane] : 0.0;
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (o < nw) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    __syncthreads();
    return t;
}

// acc[k] += f[k & 1][t] win[j + D] for output k of a chunk whose window
// element j is input position (first output - HL + j).  FP32: outputs 2m,
// 2m + 1 take one packed FMA per window element, the element broadcast and
// the two taps a pair from tp (two FMAs per lane per instruction).
template <typename T, int KIND, int NOUT, int D, int NW>
__device__ __forceinline__ void fir(const T (&win)[NW], const T (&f)[2][32],
                                    const float2 (&tp)[32], T (&acc)[NOUT]) {
    constexpr int NT = KT<KIND>::NT;
    constexpr int W = NOUT + NT - 1 + KT<KIND>::EXTRA;
    if constexpr (sizeof(T) == 4) {
        static_assert(NOUT % 2 == 0, "output pairs");
        float2 a2[NOUT / 2];
        #pragma unroll
        for (int m = 0; m < NOUT / 2; ++m) a2[m] = make_float2(acc[2 * m], acc[2 * m + 1]);
        static_for<W>([&](auto jc) {
            constexpr int j = decltype(jc)::value;
            const float2 ww = make_float2(win[j + D], win[j + D]);
            static_for<NOUT / 2>([&](auto mc) {
                constexpr int d = j - 2 * decltype(mc)::value;
                if constexpr (pair_on<KIND>(d))
                    a2[decltype(mc)::value] = __ffma2_rn(tp[d], ww, a2[decltype(mc)::value]);
            });
        });
        #pragma unroll
        for (int m = 0; m < NOUT / 2; ++m) {
            acc[2 * m] = a2[m].x;
            acc[2 * m + 1] = a2[m].y;
        }
    } else {
        static_for<W>([&](auto jc) {
            constexpr int j = decltype(jc)::value;
            static_for<NOUT>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                constexpr int t = j - k - ((k & 1) ? KT<KIND>::OFF1 : KT<KIND>::OFF0);
                if constexpr (tap_on<KIND>(t)) acc[k] = fma(f[k & 1][t], win[j + D], acc[k]);
            });
        });
    }
}

}  // namespace
}  // namespace wvl
