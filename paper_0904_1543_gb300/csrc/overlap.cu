// Orbital scalar products in compressed form.  The wavelet basis is
// orthonormal (Sec. "Daubechies basis and wavelet transformation": the
// scaling functions and wavelets of Eq. wavef0 are orthonormal, so the scalar
// product of two orbitals is the sum of the products of their coefficients,
// taken directly on the compressed vectors).
//
// S[i][j] = sum_k a_i[k] b_j[k] for blocks of orbitals (overlap_mma.cu), and the
// per-orbital products of wvl_dot here: both accurate to FP64 whatever the
// coefficients' precision, by fixed-order two-stage reductions.
#include <algorithm>
#include <cstdint>

#include <cuda_runtime.h>

#include "dot_acc.cuh"
#include "wvl.h"
#include "wvl_internal.h"

namespace wvl {
namespace {

// FP32 terms (k = t0, t0 + step, ..) whose products left the range of the split (dot_acc.cuh),
// or are all zero: once more on other scales, 2^96 up or down, and only what that does
// not reach either in FP64 (a whole call on 256 rows of 884736 coefficients: 308 us in range,
// 429 of 1e-12 and 421 of zeros, which straight to FP64 take 1366 and without the split 1269).
// Inline and not unrolled, so that the kernel keeps five blocks per SM (three: 440 in range).
__device__ __forceinline__ double dot_rescan(const float* x, const float* y, long long t0, long long end,
                                          long long step, bool vec, bool up) {
    const float2 sc = up ? make_float2(0x1p48f, 0x1p48f) : make_float2(0x1p-48f, 0x1p-48f);
    DotAcc<float> acc;
    float both = 0.f;   // largest of the terms' smaller factors: 0 if every term has a zero
    auto add = [&](float2 u, float2 v) {
        u = __fmul2_rn(u, sc);
        v = __fmul2_rn(v, sc);
        acc.add(u, v);
        both = fmaxf(both, fmaxf(fminf(fabsf(u.x), fabsf(v.x)), fminf(fabsf(u.y), fabsf(v.y))));
    };
    if (vec) {
        #pragma unroll 1
        for (long long k = t0; k < end; k += step) {
            const float4 u = __ldg(reinterpret_cast<const float4*>(x) + k);
            const float4 v = __ldg(reinterpret_cast<const float4*>(y) + k);
            add(make_float2(u.x, u.y), make_float2(v.x, v.y));
            add(make_float2(u.z, u.w), make_float2(v.z, v.w));
        }
    } else {
        #pragma unroll 1
        for (long long k = t0; k < end; k += step) add(make_float2(x[k], 0.f), make_float2(y[k], 0.f));
    }
    if (acc.ok()) return acc.get() * (up ? 0x1p-96 : 0x1p96);
    if (up && both == 0.f && acc.pmax == 0.f && isfinite(acc.s.x) && isfinite(acc.s.y)) return 0.0;
    double s = 0.0;
    const int per = vec ? 4 : 1;
    for (long long k = t0; k < end; k += step)
        for (int q = 0; q < per; ++q) s = fma((double)x[k * per + q], (double)y[k * per + q], s);
    return s;
}

// d[o] partials: block b of orbital o sums a[o][k] b[o][k] over its k.  Rows of
// whole 16-byte words are read as such (four of each row in flight); FP32 terms
// are summed as in dot_acc.cuh (FP64 conversions and FMAs per term kept the FP64
// pipe full: 1270 us for 256 orbitals of 884736 coefficients, 265 us now).
template <typename T>
__global__ void __launch_bounds__(256, 5) dot_part_kernel(const T* __restrict__ a,
                                                       const T* __restrict__ b, long long len,
                                                       double* __restrict__ part) {
    __shared__ double red[8];
    const int o = blockIdx.y;
    const T* x = a + (long long)o * len;
    const T* y = b + (long long)o * len;
    constexpr int PER = 16 / (int)sizeof(T);
    const bool vec = len % PER == 0;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long step = (long long)gridDim.x * blockDim.x;
    DotAcc<T> acc;
    if (vec) {
        #pragma unroll 4
        for (long long k = t0; k < len / PER; k += step) {
            if constexpr (sizeof(T) == 4) {
                const float4 u = __ldg(reinterpret_cast<const float4*>(x) + k);
                const float4 v = __ldg(reinterpret_cast<const float4*>(y) + k);
                acc.add(make_float2(u.x, u.y), make_float2(v.x, v.y));
                acc.add(make_float2(u.z, u.w), make_float2(v.z, v.w));
            } else {
                const double2 u = __ldg(reinterpret_cast<const double2*>(x) + k);
                const double2 v = __ldg(reinterpret_cast<const double2*>(y) + k);
                acc.add(u.x, v.x);
                acc.add(u.y, v.y);
            }
        }
    } else {
        #pragma unroll 4
        for (long long k = t0; k < len; k += step) acc.add(x[k], y[k]);
    }
    double s = acc.get();
    if constexpr (sizeof(T) == 4)
        if (!acc.ok()) s = dot_rescan(x, y, t0, vec ? len / PER : len, step, vec, acc.pmax < 1.f);
    #pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        part[(long long)o * gridDim.x + blockIdx.x] = t;
    }
}

constexpr int DOT_BLOCKS = 64;   // most partials per orbital of wvl_dot

}  // namespace
}  // namespace wvl

using namespace wvl;

namespace {
wvl_status ov_fail(wvl_status s, const char* msg) { return set_error(s, msg); }
bool misaligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) != 0; }
bool bad_prec(int prec) { return prec != WVL_F64 && prec != WVL_F32 && prec != WVL_F64_EMU; }
}  // namespace

extern "C" wvl_status wvl_overlap_workspace_size(int prec, int na, int nb, long long len,
                                                 size_t* bytes) {
    clear_error();
    if (!bytes) return ov_fail(WVL_EINVAL, "bytes is NULL");
    if (bad_prec(prec)) return ov_fail(WVL_EINVAL, "prec must be WVL_F64, WVL_F32 or WVL_F64_EMU");
    if (na < 0 || nb < 0 || len < 0) return ov_fail(WVL_EINVAL, "negative size");
    const int a1 = std::max(na, 1), b1 = std::max(nb, 1);
    const long long l1 = std::max(len, 1LL);
    const size_t ov = overlap_mma_ws_bound(a1, b1, l1);
    const size_t dot = (size_t)std::max(na, 1) * DOT_BLOCKS * sizeof(double);
    *bytes = std::max(ov, dot);
    return WVL_OK;
}

extern "C" wvl_status wvl_overlap(int prec, int na, const void* a, int nb, const void* b,
                                  long long len, double* S, void* ws, size_t ws_bytes,
                                  void* stream) {
    clear_error();
    if (bad_prec(prec)) return ov_fail(WVL_EINVAL, "prec must be WVL_F64, WVL_F32 or WVL_F64_EMU");
    if (na < 0 || nb < 0 || len < 0) return ov_fail(WVL_EINVAL, "negative size");
    if (na == 0 || nb == 0) return WVL_OK;
    if (!a || !b || !S || !ws) return ov_fail(WVL_EINVAL, "a, b, S and ws must not be NULL");
    if (misaligned(a) || misaligned(b) || misaligned(S) || misaligned(ws))
        return ov_fail(WVL_EINVAL, "a, b, S and ws must be 16-byte aligned");
    if (na > (1 << 20) || nb > (1 << 20)) return ov_fail(WVL_EUNSUPPORTED, "too many orbitals");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool sym = (a == b) && (na == nb);
    // the largest overlaps taken: 65535 blocks of 32 x 32 entries (when symmetric, on
    // and above the diagonal)
    const long long ti = (na + 31) / 32, tj = (nb + 31) / 32;
    if ((sym ? ti * (ti + 1) / 2 : ti * tj) > 65535) return ov_fail(WVL_EUNSUPPORTED, "too many tiles");
    if (ws_bytes < overlap_mma_ws(na, nb, len, sym))
        return ov_fail(WVL_ENOMEM_WS, "workspace smaller than wvl_overlap_workspace_size()");
    cudaError_t e = launch_overlap_mma(prec, na, a, nb, b, len, sym, S, ws, st);
    return e == cudaSuccess ? WVL_OK : ov_fail(WVL_ECUDA, cudaGetErrorString(e));
}

extern "C" wvl_status wvl_dot(int prec, int n, const void* a, const void* b, long long len,
                              double* d, void* ws, size_t ws_bytes, void* stream) {
    clear_error();
    if (bad_prec(prec)) return ov_fail(WVL_EINVAL, "prec must be WVL_F64, WVL_F32 or WVL_F64_EMU");
    if (n < 0 || len < 0) return ov_fail(WVL_EINVAL, "negative size");
    if (n == 0) return WVL_OK;
    if (!a || !b || !d || !ws) return ov_fail(WVL_EINVAL, "a, b, d and ws must not be NULL");
    if (misaligned(a) || misaligned(b) || misaligned(d) || misaligned(ws))
        return ov_fail(WVL_EINVAL, "a, b, d and ws must be 16-byte aligned");
    if (n > 65535) return ov_fail(WVL_EUNSUPPORTED, "more than 65535 orbitals");
    if (ws_bytes < (size_t)n * DOT_BLOCKS * sizeof(double))
        return ov_fail(WVL_ENOMEM_WS, "workspace smaller than wvl_overlap_workspace_size()");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double* part = static_cast<double*>(ws);
    // 32 terms per thread, fewer where that leaves the SMs without four blocks each: a
    // thread's end (six conversions, five FP64 additions in the FP32 form) is worth
    // several terms
    const long long want = std::max((len + 8191) / 8192,
                                    std::min((608LL + n - 1) / n, (len + 1023) / 1024));
    const int blocks = (int)std::max(1LL, std::min<long long>(want, DOT_BLOCKS));
    const dim3 grid((unsigned)blocks, (unsigned)n);
    if (prec == WVL_F32)
        dot_part_kernel<float><<<grid, 256, 0, st>>>(static_cast<const float*>(a),
                                                     static_cast<const float*>(b), len, part);
    else
        dot_part_kernel<double><<<grid, 256, 0, st>>>(static_cast<const double*>(a),
                                                      static_cast<const double*>(b), len, part);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return ov_fail(WVL_ECUDA, cudaGetErrorString(e));
    e = launch_reduce_parts(part, nullptr, blocks, n, d, st);
    return e == cudaSuccess ? WVL_OK : ov_fail(WVL_ECUDA, cudaGetErrorString(e));
}
