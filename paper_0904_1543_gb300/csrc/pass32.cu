// The FP32 passes that read or write the compressed form and the potential pass: the
// first synthesis pass, the last analysis pass and magic-filter pass 3 (Eqs. 1dconvtrans).
// The others run in pass_kernel.cuh.
//
// A CTA takes a tile of LT lines (8 to 32) of one orbital and keeps them transposed in
// shared memory: row j holds input position j - HL of every line of the tile, the
// wrapped halos being rows of their own.  A thread computes 8 consecutive outputs
// of 4 neighbouring lines: a window row is one 16-byte word per thread, whose two
// halves are the operands of packed FMAs (two lines per lane and instruction, the
// tap broadcast), and an output row is one 16-byte word, as the lines run fastest in
// the output.  Lines are read 16 (or 8, where only that is aligned) bytes at a time,
// by 16 (8) lines x 2 (4) words per warp, so that whole sectors are read and the
// transposed words of a warp fall on distinct banks.
//
// On the full grid the tiles of the compressed passes take the same range of lines of
// two neighbouring rows (both values of the parity that is not along the line), so
// that all eight components of a coarse point are in the tile: records of seven wavelet
// coefficients are read and written whole, consecutive lanes on consecutive addresses,
// through shared memory.  The row-wise kernel copies them element by element, at two and
// a half times the time of a plain pass.  The potential pass gains from 16-byte accesses to V
// and its outputs and from shared memory for density sums only where there is a density
// (a CTA without holds half as much, so twice as many fit); an instance per kind of grid and
// density keeps only its own state.  Microseconds for 64 orbitals
// on a coarse 40^3 cell (32.8 M points, 39 at the copy rate), row-wise and here: synthesis
// pass 1 140 / 102, analysis pass 3 138 / 90; on 37x45x51 the potential pass takes 488 / 200
// without a density and 568 / 268 with one, 48 orbitals there in the other two 139 / 104 and
// 160 / 122.  Small calls stay with the row-wise kernel (use_pass32).  Plain and kinetic passes stay
// with the row-wise kernel: 56 against 66, as its lines arrive by asynchronous copies while
// other CTAs of the SM (fewer registers, more of them) compute.
//
// Sums are in the order of the taps, as in the row-wise kernel: the same bits.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include <cuda_runtime.h>

#include "pass_kernel.cuh"
#include "static_for.cuh"

namespace wvl {
namespace {

constexpr int P32_R = 8;          // outputs per thread and line
constexpr int P32_THREADS = 256;  // most threads per CTA
constexpr int P32_SMEM = 200 * 1024;
// CTAs of the most threads that an SM's registers are split for: three (80 registers) in the
// compressed passes; two (128) in the potential pass, which spills 404 bytes at 80 and whose
// CTAs have 32 to 128 threads (64 orbitals with density on a free 16^3 box, in the same
// groups: 172 us at 80, 116 at 128; on a periodic 37x45x51 cell 364 and 274)
__host__ __device__ constexpr int p32_ctas(int mode) { return mode == M_POT ? 2 : 3; }

__host__ __device__ constexpr int p32_ltp(int LT) { return LT + 4; }   // row stride, 16-byte rows
// rows of the tile: the windows of ceil(n / 8) chunks
template <int KIND>
__host__ __device__ constexpr int p32_rows(int n) {
    return (n + P32_R - 1) / P32_R * P32_R + KT<KIND>::NT - 1 + KT<KIND>::EXTRA;
}

// values per word that an array's address allows: a caller's may start anywhere
__device__ __forceinline__ int p32_words(const float* p) {
    const unsigned b = (unsigned)reinterpret_cast<unsigned long long>(p);
    return (b & 15) == 0 ? 4 : (b & 7) == 0 ? 2 : 1;
}

// four values at p in words of w values (4, 2 or 1: what every address of the column
// allows), the first nv of them only
__device__ __forceinline__ void store4(float* p, float4 v, int nv, int w) {
    if (w == 4) {
        *reinterpret_cast<float4*>(p) = v;
    } else if (w == 2) {
        reinterpret_cast<float2*>(p)[0] = make_float2(v.x, v.y);
        reinterpret_cast<float2*>(p)[1] = make_float2(v.z, v.w);
    } else {
        p[0] = v.x;
        if (nv > 1) p[1] = v.y;
        if (nv > 2) p[2] = v.z;
        if (nv > 3) p[3] = v.w;
    }
}
__device__ __forceinline__ float4 load4(const float* p, int nv, int w) {
    if (w == 4) return *reinterpret_cast<const float4*>(p);
    if (w == 2) {
        const float2 a = reinterpret_cast<const float2*>(p)[0], b = reinterpret_cast<const float2*>(p)[1];
        return make_float4(a.x, a.y, b.x, b.y);
    }
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    v.x = p[0];
    if (nv > 1) v.y = p[1];
    if (nv > 2) v.z = p[2];
    if (nv > 3) v.w = p[3];
    return v;
}

template <int V> struct VecOf;
template <> struct VecOf<1> { using T = float; };
template <> struct VecOf<2> { using T = float2; };
template <> struct VecOf<4> { using T = float4; };

// The tile's lines: line l is line at(l) of the orbital, valid(l) tells whether it exists.
struct Tile {
    int a0, lt;          // plain: lines a0 .. a0 + lt - 1
    bool pairs;          // two runs of h lines: x0 .. of rows 2 pp and 2 pp + 1 of M1 lines
    int h, x0, nvh, r0, M1;
    __device__ __forceinline__ int at(int l) const {
        return pairs ? (r0 + (l >= h)) * M1 + x0 + (l >= h ? l - h : l) : a0 + l;
    }
    __device__ __forceinline__ bool valid(int l) const { return pairs ? (l >= h ? l - h : l) < nvh : l < lt; }
    // of the four lines from l (a multiple of 4)
    __device__ __forceinline__ int nvalid(int l) const {
        return max(0, min(4, (pairs ? nvh - (l >= h ? l - h : l) : lt - l)));
    }
};

// nsrc elements of every line of the tile, element x to row x + d of dst; rows outside
// [0, rows) are left out
template <int V>
__device__ __forceinline__ void stage_lines(const Tile& t, const float* __restrict__ in, int nsrc, int d,
                                            int rows, float* __restrict__ dst, int LT) {
    using W = typename VecOf<V>::T;
    const int LTP = p32_ltp(LT);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    const int LL = min(4 * V, LT), PP = 32 / LL;   // lines x words per warp
    const int ll = lane & (LL - 1), pl = lane / LL;
    const int nq = nsrc / V, dq = nw * PP;
    constexpr int U = 4;
    #pragma unroll 1
    for (int l = ll; l < LT; l += LL) {
        if (!t.valid(l)) continue;
        const W* __restrict__ src = reinterpret_cast<const W*>(in + (long long)t.at(l) * nsrc);
        #pragma unroll 1
        for (int q0 = warp * PP + pl; q0 < nq; q0 += U * dq) {
            W v[U];
            #pragma unroll
            for (int u = 0; u < U; ++u)
                if (q0 + u * dq < nq) v[u] = __ldg(src + q0 + u * dq);
            #pragma unroll
            for (int u = 0; u < U; ++u) {
                if (q0 + u * dq >= nq) break;
                const float* e = reinterpret_cast<const float*>(&v[u]);
                const int j = (q0 + u * dq) * V + d;
                float* const s = dst + j * LTP + l;
                if (j >= 0 && j + V <= rows) {
                    #pragma unroll
                    for (int k = 0; k < V; ++k) s[k * LTP] = e[k];
                } else {
                    #pragma unroll
                    for (int k = 0; k < V; ++k)
                        if (j + k >= 0 && j + k < rows) s[k * LTP] = e[k];
                }
            }
        }
    }
}
// the halo rows of periodic lines, from the rows of the same positions
__device__ __forceinline__ void wrap_rows(float* X, int n, int HL, int rows, int LT) {
    const int LTP = p32_ltp(LT), ng = LT / 4;
    const int g = threadIdx.x & (ng - 1);
    for (int k = threadIdx.x / ng; k < rows - n; k += (int)blockDim.x / ng) {
        const int r = k < HL ? k : k + n;   // halo row
        int x = r - HL;
        while (x < 0) x += n;
        while (x >= n) x -= n;
        *reinterpret_cast<float4*>(X + r * LTP + 4 * g) = *reinterpret_cast<const float4*>(X + (HL + x) * LTP + 4 * g);
    }
}
__device__ __forceinline__ void stage_any(const Tile& t, const float* in, long long per, int nsrc, int d,
                                          int rows, float* dst, int LT) {
    // (per: elements per orbital)
    const int w = p32_words(in);
    if (w == 4 && nsrc % 4 == 0 && per % 4 == 0) stage_lines<4>(t, in, nsrc, d, rows, dst, LT);
    else if (w >= 2 && nsrc % 2 == 0 && per % 2 == 0) stage_lines<2>(t, in, nsrc, d, rows, dst, LT);
    else stage_lines<1>(t, in, nsrc, d, rows, dst, LT);
}

// synthesis pass 1 on the full grid: the tile's coarse rows i3 = pp, i2 = x0 / 2 .. hold
// contiguous scaling coefficients and records of seven wavelet coefficients
__device__ __forceinline__ void stage_records(const Tile& t, const Seg<float>& S, const float* cc, int HL,
                                              float* dst, int LT) {
    const int LTP = p32_ltp(LT), n1 = S.n1;
    const int nr = t.nvh / 2;                 // coarse rows
    const long long k0 = ((long long)(t.r0 / 2) * S.n2 + t.x0 / 2) * n1;
    auto put = [&](int row, int i1, int mu, float v) {
        const int l = (mu >> 2) * t.h + 2 * row + (mu >> 1 & 1);
        const int j = HL + 2 * i1 + (mu & 1);
        dst[j * LTP + l] = v;
    };
    const int T = blockDim.x;
    {
        const float* const c0 = cc + k0;
        int row = threadIdx.x / n1, i1 = threadIdx.x - row * n1;
        for (int e = threadIdx.x; e < nr * n1; e += T) {
            put(row, i1, 0, __ldg(c0 + e));
            i1 += T;
            while (i1 >= n1) { i1 -= n1; ++row; }
        }
    }
    const float* const cf = cc + S.ncoarse + 7 * k0;
    const int dm = T % 7, di = T / 7;
    int k = threadIdx.x / 7, m = threadIdx.x - 7 * k;   // point of the rows, component - 1
    int row = k / n1, i1 = k - row * n1;
    const int total = 7 * nr * n1;
    constexpr int U = 8;
    for (int e0 = threadIdx.x; e0 < total; e0 += U * T) {
        float v[U];
        #pragma unroll
        for (int u = 0; u < U; ++u)
            if (e0 + u * T < total) v[u] = __ldg(cf + e0 + u * T);
        #pragma unroll
        for (int u = 0; u < U; ++u) {
            if (e0 + u * T < total) put(row, i1, m + 1, v[u]);
            m += dm;
            i1 += di;
            if (m >= 7) { m -= 7; ++i1; }
            while (i1 >= n1) { i1 -= n1; ++row; }
        }
    }
}

// VOWN: V and rho may live on another grid; RHO: there may be a density
template <int KIND, int MODE, bool VOWN, bool RHO>
__global__ void __launch_bounds__(P32_THREADS, p32_ctas(MODE)) pass32_kernel(const __grid_constant__ PassParams<float> p) {
    extern __shared__ __align__(16) float sm[];
    __shared__ double red[P32_THREADS / 32];
    constexpr int R = P32_R, HL = KT<KIND>::HL, NT = KT<KIND>::NT;
    constexpr int W = R + NT - 1 + KT<KIND>::EXTRA;
    constexpr bool PR = MODE != M_POT;   // tiles of two rows' lines
    int si = 0;
    const long long unit = blockIdx.x;
    #pragma unroll 1
    while (si + 1 < p.nseg && unit >= p.seg[si + 1].blk0) ++si;
    const Seg<float>& S = p.seg[si];
    const int grp = (int)((unit - S.blk0) / S.tiles), tile = (int)((unit - S.blk0) - (long long)grp * S.tiles);
    const int LT = p.LT, LTP = p32_ltp(LT), n = S.n, N = S.N;
    const int rows = p32_rows<KIND>(n), nch = (n + R - 1) / R;
    Tile t;
    t.pairs = PR;
    t.h = LT / 2;
    if (PR) {
        t.M1 = MODE == M_UNCOMP ? S.N2 : S.N1;
        const int tb = (t.M1 + t.h - 1) / t.h, pp = tile / tb;
        t.x0 = (tile - pp * tb) * t.h;
        t.nvh = min(t.h, t.M1 - t.x0);
        t.r0 = 2 * pp;
        t.a0 = t.lt = 0;
    } else {
        t.a0 = tile * LT;
        t.lt = min(LT, N - t.a0);
        t.x0 = t.nvh = t.r0 = t.M1 = 0;
    }
    float* const X = sm;                       // [rows][LTP]
    // potential pass: compensated density sums, [n][LT] high and low parts
    float* const rhi = sm + rows * LTP;
    float* const rlo = rhi + n * LT;
    const int ng = LT / 4, g = threadIdx.x & (ng - 1), slot = threadIdx.x / ng;
    const int nslots = (int)blockDim.x / ng;
    const int l0 = 4 * g, nv = t.nvalid(l0);
    const int a = t.at(l0);                    // output column of the group's first line
    // words of its stores: output I of orbital o is at o P + I N + a
    const int ow = nv < 4 ? 1 : (S.P % 4 == 0 && N % 4 == 0 && a % 4 == 0) ? 4
                              : (S.P % 2 == 0 && N % 2 == 0 && a % 2 == 0) ? 2 : 1;
    const int vw = min(ow, p32_words(S.out)), aw = MODE == M_POT ? min(ow, p32_words(S.aux)) : 1;
    const int o0 = MODE == M_POT ? grp * S.opg : grp;
    const int o1 = MODE == M_POT ? min(S.norb, o0 + S.opg) : grp + 1;

    // V and rho of output I of line l0 + k: (I + vo3) vplane + vl[k], the output's own index
    // unless they live on another grid (free lines)
    int vl[4] = {0, 0, 0, 0}, vplane = N, vo3 = 0, vn3 = 0x7fffffff;
    const bool vown = VOWN && S.vN1 > 0;
    if (vown) {
        #pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int X2 = (a + k) / S.N1, X1 = (a + k) - X2 * S.N1;
            int w1 = X1 + S.vo1, w2 = X2 + S.vo2;
            if (w1 >= S.vN1) w1 -= S.vN1;
            if (w2 >= S.vN2) w2 -= S.vN2;
            vl[k] = w2 * S.vN1 + w1;
        }
        vplane = S.vN1 * S.vN2;
        vo3 = S.vo3;
        vn3 = S.vN3;
    }
    double* const rho_out = RHO ? S.rho : nullptr;

    #pragma unroll 1
    for (int orb = o0; orb < o1; ++orb) {
        if (MODE == M_POT && orb > o0) __syncthreads();   // the tile is rewritten
        // ------------------------------------------------------- staging
        if (MODE == M_UNCOMP) {
            const float* const cc = S.in + (long long)orb * S.clen;
            stage_records(t, S, cc, HL, X, LT);
        } else if (S.nin > 0) {
            // free lines: zero outside the input's interval
            const int d = HL - S.inoff;
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            float4* const X4 = reinterpret_cast<float4*>(X);
            for (int e = threadIdx.x; e < min(max(d, 0), rows) * LTP / 4; e += blockDim.x) X4[e] = z;
            for (int e = max(d + S.nin, 0) * LTP / 4 + threadIdx.x; e < rows * LTP / 4; e += blockDim.x) X4[e] = z;
            stage_any(t, S.in + (long long)orb * S.Pin, S.Pin, S.nin, d, rows, X, LT);
        } else {
            stage_any(t, S.in + (long long)orb * S.P, S.P, n, HL, rows, X, LT);
        }
        __syncthreads();
        if (S.nin == 0) {
            wrap_rows(X, n, HL, rows, LT);
            __syncthreads();
        }

        // ------------------------------------------------------ computing
        const long long obase = (long long)orb * S.P;
        const float occ = MODE == M_POT ? (float)(S.occ ? S.occ[orb] : 1.0) : 0.f;
        float osc = 1.f;
        if (MODE == M_COMP && S.gscale != nullptr) osc = (float)(2.0 * S.occ[orb] * S.gscale[0]);
        double e = 0.0;
        // full-grid compression: the results replace the tile (or go behind it where a thread
        // has several chunks)
        const bool one = nch <= nslots;
        float* const Z = one ? X : X + rows * LTP;
        #pragma unroll 1
        for (int c = slot; c < nch || (MODE == M_COMP && one && c == slot); c += nslots) {
            const int i0 = c * R;
            float2 acc[R][2];
            const bool on = c < nch;
            if (on) {
                const float* const win = X + i0 * LTP + l0;
                #pragma unroll
                for (int r = 0; r < R; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
                static_for<W>([&](auto jc) {
                    constexpr int j = decltype(jc)::value;
                    const float4 q = *reinterpret_cast<const float4*>(win + j * LTP);
                    const float2 q0 = make_float2(q.x, q.y), q1 = make_float2(q.z, q.w);
                    static_for<R>([&](auto rc) {
                        constexpr int r = decltype(rc)::value;
                        constexpr int k = j - r - ((r & 1) ? KT<KIND>::OFF1 : KT<KIND>::OFF0);
                        if constexpr (tap_on<KIND>(k)) {
                            const float2 f = make_float2(p.f[r & 1][k], p.f[r & 1][k]);
                            acc[r][0] = __ffma2_rn(f, q0, acc[r][0]);
                            acc[r][1] = __ffma2_rn(f, q1, acc[r][1]);
                        }
                    });
                });
            }
            if (MODE == M_COMP) {
                if (one) __syncthreads();   // every window was read
                if (on)
                    #pragma unroll
                    for (int r = 0; r < R; ++r)
                        if (i0 + r < n)
                            *reinterpret_cast<float4*>(Z + (i0 + r) * LTP + l0) =
                                make_float4(acc[r][0].x * osc, acc[r][0].y * osc, acc[r][1].x * osc, acc[r][1].y * osc);
                continue;
            }
            if (nv == 0) continue;
            float ech[4] = {0.f, 0.f, 0.f, 0.f};   // the chunk's energy terms per line, then added in FP64
            #pragma unroll
            for (int r = 0; r < R; ++r) {
                const int I = i0 + r;
                if (I >= n) break;
                const float4 v = make_float4(acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
                const long long oi = obase + (long long)I * N + a;
                if (MODE == M_UNCOMP) {
                    store4(S.out + oi, v, nv, vw);
                } else {
                    const float psi[4] = {v.x, v.y, v.z, v.w};
                    if (S.aux) {
                        float pot[4];
                        if (!vown) {
                            const float4 q = load4(S.aux + (oi - obase), nv, aw);
                            pot[0] = q.x; pot[1] = q.y; pot[2] = q.z; pot[3] = q.w;
                        } else {
                            int z = I + vo3;
                            if (z >= vn3) z -= vn3;
                            #pragma unroll
                            for (int k = 0; k < 4; ++k) pot[k] = k < nv ? S.aux[(long long)z * vplane + vl[k]] : 0.f;
                        }
                        float y[4];
                        #pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            y[k] = pot[k] * psi[k];
                            ech[k] = fmaf(y[k], psi[k], ech[k]);
                        }
                        if (S.out) store4(S.out + oi, make_float4(y[0], y[1], y[2], y[3]), nv, vw);
                    }
                    if (RHO && rho_out != nullptr) {
                        float4 h4 = make_float4(0.f, 0.f, 0.f, 0.f), w4 = h4;
                        float4* const ph = reinterpret_cast<float4*>(rhi + I * LT + l0);
                        float4* const pw = reinterpret_cast<float4*>(rlo + I * LT + l0);
                        if (orb > o0) {
                            h4 = *ph;
                            w4 = *pw;
                        }
                        FF f0{h4.x, w4.x}, f1{h4.y, w4.y}, f2{h4.z, w4.z}, f3{h4.w, w4.w};
                        ff_add(f0, occ * psi[0] * psi[0]);
                        ff_add(f1, occ * psi[1] * psi[1]);
                        ff_add(f2, occ * psi[2] * psi[2]);
                        ff_add(f3, occ * psi[3] * psi[3]);
                        *ph = make_float4(f0.hi, f1.hi, f2.hi, f3.hi);
                        *pw = make_float4(f0.lo, f1.lo, f2.lo, f3.lo);
                    }
                }
            }
            if (MODE == M_POT)
                #pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k < nv) e += (double)ech[k];
        }
        if (MODE == M_COMP) {
            // records of the tile's coarse points, per i3 a run of 7 np wavelet
            // coefficients and one of np scaling coefficients
            __syncthreads();
            const int np = t.nvh / 2;
            float* const cc = S.out + (long long)orb * S.clen;
            const long long nxy = (long long)S.n1 * S.n2;
            const long long k0 = (long long)(t.r0 / 2) * S.n1 + t.x0 / 2;
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
            // element pos of a run -> offset from row 2 i3 of Z
            int zo[2];
            #pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int pos = lane + 32 * u;
                if (pos < 7 * np) {
                    const int i1 = pos / 7, mu = pos - 7 * i1 + 1;
                    zo[u] = (mu >> 2) * LTP + (mu >> 1 & 1) * t.h + 2 * i1 + (mu & 1);
                } else {
                    zo[u] = 2 * (pos - 7 * np);
                }
            }
            for (int i3 = warp; i3 < n / 2; i3 += nw) {
                const float* const z = Z + 2 * i3 * LTP;
                const long long k = (long long)i3 * nxy + k0;
                #pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int pos = lane + 32 * u;
                    if (pos < 7 * np) cc[S.ncoarse + 7 * k + pos] = z[zo[u]];
                    else if (pos < 8 * np) cc[k + pos - 7 * np] = z[zo[u]];
                }
            }
        }
        if (MODE == M_POT && S.aux) {
            #pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
            if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
            __syncthreads();
            if (threadIdx.x == 0) {
                double s = 0.0;
                for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
                S.part[(long long)orb * S.tiles + tile] = s;
            }
        }
    }

    // the group's density, consecutive lanes on consecutive lines
    if (RHO && rho_out != nullptr) {
        __syncthreads();
        const int l = threadIdx.x & (LT - 1);
        if (l >= t.lt) return;
        long long q0 = t.a0 + l;
        if (vown) {
            const int X2 = (int)q0 / S.N1, X1 = (int)q0 - X2 * S.N1;
            int w1 = X1 + S.vo1, w2 = X2 + S.vo2;
            if (w1 >= S.vN1) w1 -= S.vN1;
            if (w2 >= S.vN2) w2 -= S.vN2;
            q0 = (long long)w2 * S.vN1 + w1;
        }
        double* const rho = rho_out + (S.rho_gstride == 0 ? 0 : grp * S.rho_gstride) + q0;
        #pragma unroll 2
        for (int I = threadIdx.x / LT; I < n; I += blockDim.x / LT) {
            int z = I + vo3;
            if (z >= vn3) z -= vn3;
            const double v = (double)rhi[I * LT + l] + (double)rlo[I * LT + l];
            double* const q = rho + (long long)z * vplane;
            *q = S.rho_gstride == 0 ? *q + v : v;
        }
    }
}

template <int KIND, int MODE, bool VOWN, bool RHO>
cudaError_t p32_attr() {
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(done.load() & bit)) {
        err = cudaFuncSetAttribute((pass32_kernel<KIND, MODE, VOWN, RHO>), cudaFuncAttributeMaxDynamicSharedMemorySize, P32_SMEM);
        if (err != cudaSuccess) return err;
        done.fetch_or(bit);
    }
    return cudaSuccess;
}

// f(kind, mode, V and rho on another grid, density) of every instance
template <typename F>
void for_each_p32(F&& f) {
    using std::integral_constant;
#define P32_K(kind, mode, vown, rho) \
    f(integral_constant<int, kind>{}, integral_constant<int, mode>{}, std::vown##_type{}, std::rho##_type{})
    P32_K(K_SYN, M_UNCOMP, false, false);
    P32_K(K_ANA, M_COMP, false, false);
    P32_K(K_MF, M_POT, false, false);
    P32_K(K_MF, M_POT, false, true);
    P32_K(K_MF, M_POT, true, false);
    P32_K(K_MF, M_POT, true, true);
#undef P32_K
}

}  // namespace

int pass32_threads(int LT, int nmax) {
    const int items = LT / 4 * ((nmax + P32_R - 1) / P32_R);
    return std::max(32, std::min((items + 31) / 32 * 32, P32_THREADS));
}

int pass32_ctas(int threads, size_t smem) {   // (1100: the static part)
    return (int)std::max<size_t>(1, std::min<size_t>(227 * 1024 / (smem + 1100), 512 / threads));
}

size_t pass32_smem(int kind, int mode, int LT, int n, bool rho) {
    const size_t rows = kind == K_SYN ? p32_rows<K_SYN>(n) : kind == K_ANA ? p32_rows<K_ANA>(n) : p32_rows<K_MF>(n);
    const size_t nch = (n + P32_R - 1) / P32_R;
    size_t b = rows * p32_ltp(LT);
    if (mode == M_POT && rho) b += 2 * (size_t)n * LT;
    // the compression's results behind the tile where a thread has several chunks
    if (mode == M_COMP && (long long)nch * (LT / 4) > P32_THREADS) b += (size_t)n * p32_ltp(LT);
    return b * sizeof(float);
}

cudaError_t launch_pass32(int kind, int mode, const PassParams<float>& p, long long nunits, int threads,
                          size_t smem, cudaStream_t st) {
    if (nunits <= 0) return cudaSuccess;
    if (nunits > 0x7fffffffLL || smem > (size_t)P32_SMEM) return cudaErrorInvalidConfiguration;
    bool vown = false, rho = false;
    for (int k = 0; k < p.nseg; ++k) {
        vown |= mode == M_POT && p.seg[k].vN1 > 0;
        rho |= mode == M_POT && p.seg[k].rho != nullptr;
    }
    cudaError_t e = cudaErrorInvalidValue;
    for_each_p32([&](auto k, auto m, auto v, auto r) {
        if (kind != k() || mode != m() || vown != v() || rho != r()) return;
        if ((e = p32_attr<k(), m(), v(), r()>()) != cudaSuccess) return;
        pass32_kernel<k(), m(), v(), r()><<<dim3((unsigned)nunits), dim3(threads), smem, st>>>(p);
        count_launches(1);
        e = cudaGetLastError();
    });
    return e;
}

cudaError_t prepare_pass32() {
    cudaError_t e = cudaSuccess;
    for_each_p32([&](auto k, auto m, auto v, auto r) {
        if (e == cudaSuccess) e = p32_attr<k(), m(), v(), r()>();
    });
    return e;
}

}  // namespace wvl
