// The preconditioner's conjugate gradient in FP32 (paper Eq. precon) on cells whose
// xy planes fit in shared memory.
//
// The operator in the compressed basis, A = S^T (K - eps) S, separates: with
// S_d^T S_d = 1 on every axis (orthonormality of h and g, Eq. refinement),
//   A = B_1 + B_2 + B_3 - eps,   B_d = S_d^T T_d S_d,
// each B_d a 1D filter on the interleaved coefficients of axis d whose taps depend
// on the parity of the output (scaling function or wavelet): 58 taps for the 27
// of T_d.  In FP32 the 46 of offsets -22 .. 23 (even outputs) and -23 .. 22 (odd ones)
// are applied; the others add up to 2e-11 of the filter's absolute sum, 1/1500
// of the rounding of the sum they would enter.  138 FMAs per point
// instead of the 177 of synthesis, kinetic filter and analysis, and one sweep per axis
// instead of three.
//
// The vectors r, p, q, x stay in the interleaved layout [z][y][x] between the first
// kernel, which reads the compressed g, and the last, which writes the compressed x.
// Per iteration:
//   hz_plane  p = M^-1 r + beta p and x += alpha p of the iteration before, on one
//             xy plane on its way into shared memory;  w = (B_1 + B_2) p
//   hz_col    q = w + B_3 p - eps p on tiles of 32 columns, partials of p.q
//   hz_step   r -= alpha q, partials of r.z (z = M^-1 r is formed where it is used)
// 48 bytes per point and iteration, where the transposing passes and vector
// kernels moved 156.  256 orbitals on a coarse 48^3 cell, 5 iterations: 42.7 -> 10.4 ms.
//
// A thread of hz_plane owns 8 rows x 4 columns of w.  Its row sums read 13
// 16-byte words per row (wrapped offsets kept in registers), its column sums
// one per row of the window; the plane needs no second buffer and no barrier
// but the one after loading, so that up to five planes are resident per SM (80
// registers; 119 without the cap, two planes of 256 threads, 12.2 ms) and one's
// loads run under another's FMAs.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <utility>

#include <cuda_runtime.h>

#include "dot_acc.cuh"
#include "static_for.cuh"
#include "wvl_internal.h"

namespace wvl {
namespace {

constexpr int HZ_NT = 46;          // taps
constexpr int HZ_LO = 22;          // offset of the first tap: -22 (even outputs), -23 (odd)
constexpr int HZ_PAD = 24;         // wrapped rows before and after a column, at least
constexpr int HZ_RC = 8;           // rows per item
constexpr int HZ_PT = 256;         // most threads of hz_plane
constexpr int HZ_SMEM = 220 * 1024;
constexpr int HZ_MAXN = 512;       // largest extent
constexpr int HZ_CT = 32;          // columns per tile of hz_col

struct HzParams {
    float tap[3][2][48];    // B_d per axis and parity, in offset order
    float2 pair[48];        // axis 1: the taps of outputs 2m and 2m + 1 for one input
    double diag[8];         // diagonal of S^T K S per component mu
    const double* eps;
    const double* rz0;      // r.z before and after the last step, p.q of it, per orbital
    const double* rz1;
    const double* pq;
    float* r;
    float* p;
    float* q;
    float* w;
    float* x;
    double* part;
    const float* g;         // compressed right-hand side
    float* xc;              // compressed result
    long long P;
    int N1, N2, N3, norb;
    int tiles;              // hz_col: tiles per orbital
    int nblk;               // hz_step, hz_init: blocks per orbital
};

// rowoff[HZ_PAD + j] = (j mod n) * stride for j in [-HZ_PAD, nr + HZ_PAD), nr = n rounded
// up to whole items
__device__ __forceinline__ void hz_rowoff(int* rowoff, int n, int stride) {
    const int nr = (n + HZ_RC - 1) / HZ_RC * HZ_RC;
    for (int j = (int)threadIdx.x; j < nr + 2 * HZ_PAD; j += blockDim.x) {
        int m = (j - HZ_PAD) % n;
        if (m < 0) m += n;
        rowoff[j] = m * stride;
    }
}

// acc[k][.] += sum_D B[k & 1][D] src(row r0 + k + D, 4 columns at base)
__device__ __forceinline__ void hz_col_sum(const float* __restrict__ base, const int* __restrict__ ro,
                                           const float (&f)[2][48], float2 (&acc)[HZ_RC][2]) {
    // window row j is row r0 - HZ_LO + j; rows k and k + 1 (k even) both take j = k .. k + 45
    static_for<HZ_RC - 2 + HZ_NT>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        const float4 v = *reinterpret_cast<const float4*>(base + ro[j]);
        const float2 a = make_float2(v.x, v.y), b = make_float2(v.z, v.w);
        static_for<HZ_RC>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            constexpr int t = j - (k & ~1);
            if constexpr (t >= 0 && t < HZ_NT) {
                const float2 c = make_float2(f[k & 1][t], f[k & 1][t]);
                acc[k][0] = __ffma2_rn(c, a, acc[k][0]);
                acc[k][1] = __ffma2_rn(c, b, acc[k][1]);
            }
        });
    });
}

// 1 / (d_mu - eps_o), mu = a1 + 2 a2 + 4 a3, in shared memory
__device__ __forceinline__ void hz_minv(const HzParams& h, int o, float* minv) {
    if (threadIdx.x < 8) minv[threadIdx.x] = (float)(1.0 / (h.diag[threadIdx.x] - h.eps[o]));
}

// The block's total of the threads' scalar-product terms (dot_acc.cuh: three FP32 numbers of
// about 70 bits), in a fixed order; FP64 from the warp on (per thread, the conversions and
// additions kept hz_col's FP64 pipe busy for a third of its time).  wide: the FP64 sum of a
// thread whose terms left the range of the split.
__device__ __forceinline__ float hz_two_sum(float& a, float x) {
    const float t = a + x, b = t - a, e = (a - (t - b)) + (x - b);
    a = t;
    return e;
}
__device__ __forceinline__ void hz_add3(float (&v)[3], float h, float m, float l) {
    const float e = hz_two_sum(v[0], h);
    const float e1 = hz_two_sum(v[1], m), e2 = hz_two_sum(v[1], e);
    v[2] += l + (e1 + e2);
}
__device__ __forceinline__ double hz_block_sum(const DotAcc<float>& d, bool on, bool ok, double wide, double* red) {
    float v[3] = {0.f, 0.f, 0.f};
    if (on && ok) {
        v[0] = d.s.x;
        v[1] = d.c.x;
        v[2] = d.d.x;
        hz_add3(v, d.s.y, d.c.y, d.d.y);
    }
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h = __shfl_down_sync(0xffffffffu, v[0], o), m = __shfl_down_sync(0xffffffffu, v[1], o);
        hz_add3(v, h, m, __shfl_down_sync(0xffffffffu, v[2], o));
    }
    double t = (double)v[0] + ((double)v[1] + (double)v[2]);
    if (__any_sync(0xffffffffu, on && !ok)) {
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) wide += __shfl_down_sync(0xffffffffu, wide, o);
        t += wide;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    return t;
}

// alpha = r.z / p.q of orbital o's last step
__device__ __forceinline__ float hz_alpha(const HzParams& h, int o) { return (float)(h.rz0[o] / h.pq[o]); }

// 16-byte word v of an orbital's [z][y][x] array -> 2 a2 + 4 a3 of its row
__device__ __forceinline__ int hz_mu(int v, int ncv, int N2) {
    const int row = v / ncv;
    const int z = row / N2;
    return 2 * ((row - z * N2) & 1) + 4 * (z & 1);
}

// r = g in the interleaved layout; partials of g.M^-1 g.  A thread takes a coarse
// point: its scaling coefficient and its record of seven wavelet coefficients.
__global__ void __launch_bounds__(256) hz_init_kernel(const __grid_constant__ HzParams h) {
    __shared__ float minv[8];
    __shared__ double red[8];
    const int o = blockIdx.y;
    hz_minv(h, o, minv);
    __syncthreads();
    const int n1 = h.N1 / 2, n2 = h.N2 / 2, m = (int)(h.P / 8);
    const float* const gc = h.g + (long long)o * h.P;
    float* const r = h.r + (long long)o * h.P;
    DotAcc<float> acc;
    for (int k = blockIdx.x * 256 + threadIdx.x; k < m; k += gridDim.x * 256) {
        const int row = k / n1, i1 = k - row * n1;
        const int i3 = row / n2, i2 = row - i3 * n2;
        float c[8];
        c[0] = gc[k];
        #pragma unroll
        for (int mu = 1; mu < 8; ++mu) c[mu] = gc[m + 7LL * k + mu - 1];
        #pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float2 v = make_float2(c[2 * a], c[2 * a + 1]);
            *reinterpret_cast<float2*>(
                r + ((long long)(2 * i3 + (a >> 1)) * h.N2 + 2 * i2 + (a & 1)) * h.N1 + 2 * i1) = v;
            acc.add(v, make_float2(minv[2 * a] * v.x, minv[2 * a + 1] * v.y));
        }
    }
    double s = 0.0;
    const bool ok = acc.ok();
    if (!ok) {
        for (int k = blockIdx.x * 256 + threadIdx.x; k < m; k += gridDim.x * 256)
            for (int mu = 0; mu < 8; ++mu) {
                const float c = mu == 0 ? gc[k] : gc[m + 7LL * k + mu - 1];
                s = fma((double)c, (double)(minv[mu] * c), s);
            }
    }
    const double t = hz_block_sum(acc, true, ok, s, red);
    if (threadIdx.x == 0) h.part[(long long)o * h.nblk + blockIdx.x] = t;
}

// STEP 0: p = M^-1 r;  1: x = alpha p, p = M^-1 r + beta p;  2: x += alpha p, the same p
template <int STEP>
__global__ void __maxnreg__(80) hz_plane_kernel(const __grid_constant__ HzParams h) {
    extern __shared__ __align__(16) float X[];
    __shared__ float minv[8];
    __shared__ int rowoff[HZ_MAXN + HZ_RC + 2 * HZ_PAD];
    const int N1 = h.N1, N2 = h.N2, ncv = N1 / 4;
    const int o = blockIdx.x / h.N3, z = blockIdx.x - o * h.N3;
    const long long base = (long long)o * h.P + (long long)z * N1 * N2;
    hz_minv(h, o, minv);
    hz_rowoff(rowoff, N2, N1);
    float alpha = 0.f, beta = 0.f;
    if (STEP > 0) {
        alpha = hz_alpha(h, o);
        beta = (float)(h.rz1[o] / h.rz0[o]);
    }
    __syncthreads();
    #pragma unroll 4
    for (int v = threadIdx.x; v < N2 * ncv; v += blockDim.x) {
        const int mu = 2 * ((v / ncv) & 1) + 4 * (z & 1);
        const float m0 = minv[mu], m1 = minv[mu + 1];
        const float4 r = reinterpret_cast<const float4*>(h.r + base)[v];
        float4 p = make_float4(m0 * r.x, m1 * r.y, m0 * r.z, m1 * r.w);
        if (STEP > 0) {
            const float4 q = reinterpret_cast<const float4*>(h.p + base)[v];
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (STEP > 1) x = reinterpret_cast<const float4*>(h.x + base)[v];
            x.x = fmaf(alpha, q.x, x.x); x.y = fmaf(alpha, q.y, x.y);
            x.z = fmaf(alpha, q.z, x.z); x.w = fmaf(alpha, q.w, x.w);
            reinterpret_cast<float4*>(h.x + base)[v] = x;
            p.x = fmaf(beta, q.x, p.x); p.y = fmaf(beta, q.y, p.y);
            p.z = fmaf(beta, q.z, p.z); p.w = fmaf(beta, q.w, p.w);
        }
        reinterpret_cast<float4*>(h.p + base)[v] = p;
        reinterpret_cast<float4*>(X)[v] = p;
    }
    __syncthreads();
    const int nri = (N2 + HZ_RC - 1) / HZ_RC;
    #pragma unroll 1
    for (int it = threadIdx.x; it < nri * ncv; it += blockDim.x) {
        const int k0 = it / ncv, cv = it - k0 * ncv, r0 = k0 * HZ_RC;
        float2 acc[HZ_RC][2];
        #pragma unroll
        for (int k = 0; k < HZ_RC; ++k) acc[k][0] = acc[k][1] = make_float2(0.f, 0.f);
        // the window of a row: words cv - 6 .. cv + 6 (inputs 4 cv - 24 + j), wrapped
        int off[13];
        int c = cv - 6;
        while (c < 0) c += ncv;
        #pragma unroll
        for (int i = 0; i < 13; ++i) {
            off[i] = 4 * c;
            if (++c == ncv) c = 0;
        }
        static_for<HZ_RC>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            const float* const row = X + rowoff[HZ_PAD + r0 + k];
            static_for<13>([&](auto ic) {
                constexpr int i = decltype(ic)::value;
                const float4 v = *reinterpret_cast<const float4*>(row + off[i]);
                const float e[4] = {v.x, v.y, v.z, v.w};
                // outputs 2m, 2m + 1 take input j with the pair j - 2m - 2
                static_for<8>([&](auto jm) {
                    constexpr int j = 4 * i + decltype(jm)::value / 2, m = decltype(jm)::value % 2;
                    constexpr int t = j - 2 * m - 2;
                    if constexpr (t >= 0 && t < HZ_NT)
                        acc[k][m] = __ffma2_rn(h.pair[t], make_float2(e[j & 3], e[j & 3]), acc[k][m]);
                });
            });
        });
        hz_col_sum(X + 4 * cv, rowoff + HZ_PAD + r0 - HZ_LO, h.tap[1], acc);
        float* const w = h.w + base + 4 * cv;
        #pragma unroll
        for (int k = 0; k < HZ_RC; ++k)
            if (r0 + k < N2)
                *reinterpret_cast<float4*>(w + (long long)(r0 + k) * N1) =
                    make_float4(acc[k][0].x, acc[k][0].y, acc[k][1].x, acc[k][1].y);
    }
}

// q = w + B_3 p - eps p on the tile's columns; partial of p.q.  One item (8 rows of a
// 16-byte column) per thread; w is read into the sums under the tile's copies.
__global__ void hz_col_kernel(const __grid_constant__ HzParams h) {
    extern __shared__ __align__(16) float X[];
    __shared__ double red[16];
    __shared__ int rowoff[HZ_MAXN + HZ_RC + 2 * HZ_PAD];
    const int o = blockIdx.y, N3 = h.N3;
    const int plane = h.N1 * h.N2, c0 = blockIdx.x * HZ_CT;
    const int ncv = min(HZ_CT, plane - c0) / 4;
    const float* const p = h.p + (long long)o * h.P + c0;
    const int cv = threadIdx.x & 7, r0 = (threadIdx.x >> 3) * HZ_RC;
    const bool on = cv < ncv && r0 < N3;
    if (cv < ncv)
        for (int z = threadIdx.x >> 3; z < N3; z += blockDim.x >> 3) {
            const unsigned s = (unsigned)__cvta_generic_to_shared(X + z * HZ_CT + 4 * cv);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s),
                         "l"(p + (long long)z * plane + 4 * cv) : "memory");
        }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    hz_rowoff(rowoff, N3, HZ_CT);
    float2 acc[HZ_RC][2];
    const long long qb = (long long)o * h.P + c0 + 4 * cv;
    #pragma unroll
    for (int k = 0; k < HZ_RC; ++k) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (on && r0 + k < N3) v = *reinterpret_cast<const float4*>(h.w + qb + (long long)(r0 + k) * plane);
        acc[k][0] = make_float2(v.x, v.y);
        acc[k][1] = make_float2(v.z, v.w);
    }
    const float me = (float)(-h.eps[o]);
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    double s = 0.0;
    bool ok = true;
    DotAcc<float> dot;
    if (on) {
        hz_col_sum(X + 4 * cv, rowoff + HZ_PAD + r0 - HZ_LO, h.tap[2], acc);
        #pragma unroll
        for (int k = 0; k < HZ_RC; ++k) {
            if (r0 + k >= N3) break;
            const float4 v = *reinterpret_cast<const float4*>(X + (r0 + k) * HZ_CT + 4 * cv);
            acc[k][0] = __ffma2_rn(make_float2(me, me), make_float2(v.x, v.y), acc[k][0]);
            acc[k][1] = __ffma2_rn(make_float2(me, me), make_float2(v.z, v.w), acc[k][1]);
            dot.add(make_float2(v.x, v.y), acc[k][0]);
            dot.add(make_float2(v.z, v.w), acc[k][1]);
            *reinterpret_cast<float4*>(h.q + qb + (long long)(r0 + k) * plane) =
                make_float4(acc[k][0].x, acc[k][0].y, acc[k][1].x, acc[k][1].y);
        }
        ok = dot.ok();
        if (!ok) {
            for (int k = 0; k < HZ_RC && r0 + k < N3; ++k)
                for (int e = 0; e < 4; ++e)
                    s = fma((double)X[(r0 + k) * HZ_CT + 4 * cv + e],
                            (double)h.q[qb + (long long)(r0 + k) * plane + e], s);
        }
    }
    const double t = hz_block_sum(dot, on, ok, s, red);
    if (threadIdx.x == 0) h.part[(long long)o * h.tiles + blockIdx.x] = t;
}

// r -= alpha q; partials of r.M^-1 r, or of r.r (RR)
template <bool RR>
__global__ void __launch_bounds__(256) hz_step_kernel(const __grid_constant__ HzParams h) {
    __shared__ float minv[8];
    __shared__ double red[8];
    const int o = blockIdx.y, ncv = h.N1 / 4, nv = (int)(h.P / 4);
    hz_minv(h, o, minv);
    const float ma = -hz_alpha(h, o);
    __syncthreads();
    float4* const r4 = reinterpret_cast<float4*>(h.r + (long long)o * h.P);
    const float4* const q4 = reinterpret_cast<const float4*>(h.q + (long long)o * h.P);
    DotAcc<float> acc;
    #pragma unroll 4
    for (int v = blockIdx.x * 256 + threadIdx.x; v < nv; v += gridDim.x * 256) {
        const int mu = hz_mu(v, ncv, h.N2);
        const float m0 = RR ? 1.f : minv[mu], m1 = RR ? 1.f : minv[mu + 1];
        float4 r = r4[v];
        const float4 q = q4[v];
        r.x = fmaf(ma, q.x, r.x); r.y = fmaf(ma, q.y, r.y);
        r.z = fmaf(ma, q.z, r.z); r.w = fmaf(ma, q.w, r.w);
        r4[v] = r;
        acc.add(make_float2(r.x, r.y), make_float2(m0 * r.x, m1 * r.y));
        acc.add(make_float2(r.z, r.w), make_float2(m0 * r.z, m1 * r.w));
    }
    double s = 0.0;
    const bool ok = acc.ok();
    if (!ok) {
        for (int v = blockIdx.x * 256 + threadIdx.x; v < nv; v += gridDim.x * 256) {
            const int mu = hz_mu(v, ncv, h.N2);
            const float4 r = r4[v];
            const float e[4] = {r.x, r.y, r.z, r.w};
            for (int k = 0; k < 4; ++k)
                s = fma((double)e[k], (double)((RR ? 1.f : minv[mu + (k & 1)]) * e[k]), s);
        }
    }
    const double t = hz_block_sum(acc, true, ok, s, red);
    if (threadIdx.x == 0) h.part[(long long)o * h.nblk + blockIdx.x] = t;
}

// x = (x +) alpha p, written compressed
template <bool FIRST>
__global__ void __launch_bounds__(256) hz_final_kernel(const __grid_constant__ HzParams h) {
    const int o = blockIdx.y;
    const int n1 = h.N1 / 2, n2 = h.N2 / 2, m = (int)(h.P / 8);
    const float alpha = hz_alpha(h, o);
    const long long base = (long long)o * h.P;
    float* const xc = h.xc + base;
    for (int k = blockIdx.x * 256 + threadIdx.x; k < m; k += gridDim.x * 256) {
        const int row = k / n1, i1 = k - row * n1;
        const int i3 = row / n2, i2 = row - i3 * n2;
        float c[8];
        #pragma unroll
        for (int a = 0; a < 4; ++a) {
            const long long at = base + ((long long)(2 * i3 + (a >> 1)) * h.N2 + 2 * i2 + (a & 1)) * h.N1 + 2 * i1;
            const float2 p = *reinterpret_cast<const float2*>(h.p + at);
            float2 x = make_float2(0.f, 0.f);
            if (!FIRST) x = *reinterpret_cast<const float2*>(h.x + at);
            c[2 * a] = fmaf(alpha, p.x, x.x);
            c[2 * a + 1] = fmaf(alpha, p.y, x.y);
        }
        xc[k] = c[0];
        #pragma unroll
        for (int mu = 1; mu < 8; ++mu) xc[m + 7LL * k + mu - 1] = c[mu];
    }
}

// B_d for spacing 1 (T = -a / 2): tap t of parity e multiplies the input at offset
// t - HZ_LO - e
struct HzTaps {
    double b[2][HZ_NT];
    HzTaps() {
        const FilterSet& F = filters();
        const double* f[2] = {F.h, F.g};
        for (int e = 0; e < 2; ++e)
            for (int t = 0; t < HZ_NT; ++t) {
                const int d = t - HZ_LO - e;               // input position, output at e
                const int ei = (d + e) & 1, c = (d + e - ei) / 2;   // its parity and coarse point
                double s = 0.0;
                for (int i = -7; i <= 8; ++i)
                    for (int j = -7; j <= 8; ++j) {
                        const int l = i - (2 * c + j);
                        if (l >= -14 && l <= 14) s += f[e][i + 7] * (-0.5 * F.a[l + 14]) * f[ei][j + 7];
                    }
                b[e][t] = s;
            }
    }
};

cudaError_t hz_prepare() {
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load() & bit) return cudaSuccess;
    const void* k[4] = {reinterpret_cast<const void*>(hz_plane_kernel<0>),
                        reinterpret_cast<const void*>(hz_plane_kernel<1>),
                        reinterpret_cast<const void*>(hz_plane_kernel<2>),
                        reinterpret_cast<const void*>(hz_col_kernel)};
    for (const void* f : k)
        if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, HZ_SMEM)) != cudaSuccess)
            return e;
    done.fetch_or(bit);
    return cudaSuccess;
}

}  // namespace

// Rows of whole 16-byte words, an xy plane in the shared memory of one CTA, and the
// limits of the kernels' tables and launch grids.
bool helmholtz_pcg_ok(const int Nf[3], int norb) {
    return Nf[0] % 4 == 0 && (long long)Nf[0] * Nf[1] * 4 <= HZ_SMEM && Nf[1] <= HZ_MAXN &&
           Nf[2] <= HZ_MAXN && norb <= 65535 && (long long)norb * Nf[2] <= 0x7fffffffLL;
}

cudaError_t launch_helmholtz_pcg(const int Nf[3], const double hg[3], const double diag[8], int norb,
                                 const float* g, const double* eps, int ncg, float* x, double* rr,
                                 float* const buf[5], double* const scal[3], double* const part[2],
                                 cudaStream_t st) {
    static const HzTaps T;
    cudaError_t e = hz_prepare();
    if (e != cudaSuccess) return e;
    HzParams h;
    for (int a = 0; a < 3; ++a)
        for (int p = 0; p < 2; ++p)
            for (int t = 0; t < 48; ++t) h.tap[a][p][t] = t < HZ_NT ? (float)(T.b[p][t] / (hg[a] * hg[a])) : 0.f;
    for (int t = 0; t < 48; ++t) h.pair[t] = make_float2(h.tap[0][0][t], h.tap[0][1][t]);
    for (int k = 0; k < 8; ++k) h.diag[k] = diag[k];
    h.eps = eps;
    h.r = buf[0];
    h.p = buf[1];
    h.q = buf[2];
    h.w = buf[3];
    h.x = buf[4];
    h.g = g;
    h.xc = x;
    h.N1 = Nf[0];
    h.N2 = Nf[1];
    h.N3 = Nf[2];
    h.P = (long long)Nf[0] * Nf[1] * Nf[2];
    h.norb = norb;
    const int plane = h.N1 * h.N2;
    h.tiles = (plane + HZ_CT - 1) / HZ_CT;
    // vector kernels: at least four 16-byte words per thread, 64 blocks per orbital at most
    h.nblk = (int)std::max(1LL, std::min(64LL, (h.P + 4095) / 4096));
    double *rz0 = scal[0], *rz1 = scal[1], *pq = scal[2];
    const dim3 vgrid((unsigned)h.nblk, (unsigned)norb);
    const size_t psm = (size_t)plane * 4, csm = (size_t)h.N3 * HZ_CT * 4;
    const int pitems = (h.N2 + HZ_RC - 1) / HZ_RC * (h.N1 / 4);
    // whole rounds of items over at most 256 threads: 288 items of a 96^2 plane take two
    // rounds of 160 threads (five CTAs per SM; 10.4 ms on the headline case), not
    // 256 and 32 of 256 (11.2 ms) or one of 288 (two CTAs per SM, 11.8 ms)
    const int rounds = (pitems + HZ_PT - 1) / HZ_PT;
    const int pthreads = ((pitems + rounds - 1) / rounds + 31) / 32 * 32;
    const int cthreads = ((h.N3 + HZ_RC - 1) / HZ_RC * 8 + 31) / 32 * 32;
#define HZ_LAUNCHED()                                           \
    do {                                                        \
        count_launches(1);                                      \
        if ((e = cudaGetLastError()) != cudaSuccess) return e;  \
    } while (0)
    h.part = part[0];
    hz_init_kernel<<<vgrid, 256, 0, st>>>(h);
    HZ_LAUNCHED();
    if ((e = launch_reduce_parts(part[0], nullptr, h.nblk, norb, rz0, st)) != cudaSuccess) return e;
    for (int it = 0; it < ncg; ++it) {
        // rz0: r.z before the last step; rz1: after it (the one that counts now)
        h.rz0 = rz0;
        h.rz1 = rz1;
        h.pq = pq;
        const dim3 pgrid((unsigned)((long long)norb * h.N3));
        if (it == 0) hz_plane_kernel<0><<<pgrid, pthreads, psm, st>>>(h);
        else if (it == 1) hz_plane_kernel<1><<<pgrid, pthreads, psm, st>>>(h);
        else hz_plane_kernel<2><<<pgrid, pthreads, psm, st>>>(h);
        HZ_LAUNCHED();
        if (it > 0) std::swap(rz0, rz1);
        h.rz0 = rz0;
        h.part = part[1];
        hz_col_kernel<<<dim3((unsigned)h.tiles, (unsigned)norb), cthreads, csm, st>>>(h);
        HZ_LAUNCHED();
        if ((e = launch_reduce_parts(part[1], nullptr, h.tiles, norb, pq, st)) != cudaSuccess) return e;
        const bool last = it + 1 == ncg;
        if (last && rr == nullptr) break;   // nothing reads r again
        h.part = part[0];
        if (last) hz_step_kernel<true><<<vgrid, 256, 0, st>>>(h);
        else hz_step_kernel<false><<<vgrid, 256, 0, st>>>(h);
        HZ_LAUNCHED();
        if ((e = launch_reduce_parts(part[0], nullptr, h.nblk, norb, last ? rr : rz1, st)) != cudaSuccess)
            return e;
    }
    if (ncg == 1) hz_final_kernel<true><<<vgrid, 256, 0, st>>>(h);
    else hz_final_kernel<false><<<vgrid, 256, 0, st>>>(h);
    HZ_LAUNCHED();
#undef HZ_LAUNCHED
    return cudaSuccess;
}

}  // namespace wvl
