// The plane kernels of the fused chain (fused_kernel.cu) for square FP32 planes of 32, 64, 96 or
// 128 points a side: most filters are applied along the buffer's rows of 16-byte words ("line
// items": 16 consecutive outputs of two neighbouring lines per thread), the plane being
// transposed between the filters of different axes as the outputs are stored.
//
// A plane kernel is a chain of phases between barriers, each bound half by the FMA pipe and
// half by its latencies (load, window, stores), so what counts is how much of a phase
// another one covers.  The swizzled buffers need no padding, so three 96^2 planes share an SM
// (two in the general form); 128^2 planes are alone on their SM, and a CTA per SM walks
// over them with a third buffer for the next plane (fz_tplane_shape).  Two values of a row are the operands
// of a packed FMA as they are loaded; a row item has to copy each value into both
// halves.  Extents are compile-time constants, which leaves one XOR per 16-byte load of address
// arithmetic.  Microseconds of SYN3 + SKM12 / MFTA12 in the general form and here: 128^2 (48
// orbitals) 812 / 432 and 688 / 324 (746 / 388 with extents from memory), 96^2 (64) 456 /
// 219 and 388 / 209, 64^2 (128) 267 / 123 and 239 / 119, 32^2 (512) 150 / 78 and 125 / 78 (so
// MFTA12 keeps the general form there).  Also tried at 128^2, with extents from memory: items of
// four lines (256 threads: 760 / 447), T_2 as items along the contiguous axis of a transposed s
// (800 to 820), a warp of its own for the copies (1153 / 1205: one warp's copies in flight
// are too few).
//
// Filter sums and the FP32 chains of Ekin keep the order of the general form, so that an orbital's
// results do not depend on the number of planes in its call, which chooses the form and its
// threads (fz_plane_shape): H psi has the same bits, and Ekin, whose chains are added in
// compensated pairs grouped by threads, differs from 2^-48 on if at all.
// MFT_1 before MFT_2 therefore, by rows and without a transpose (128^2 324 us, with MFT_2
// first, both as line items, 331; 96^2 209 and 207).
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "fused.cuh"

namespace wvl {
namespace {

// A buffer holds a plane as [row][col], RS floats per row, one buffer after
// the other.  The 16-byte word u of row j lies at word u ^ swz(j), so that
// eight lanes find distinct banks on consecutive words of a row, on one word of eight
// consecutive rows and on one word of eight rows four apart.
//   8 i + j -> j ^ (i & 3):  bijective in the low three bits of the row and in bits 2 to 4
__device__ __forceinline__ unsigned swz(int row) { return (unsigned)((row & 7) ^ ((row >> 3) & 3)); }

__host__ __device__ constexpr int floor8(int d) { return d >= 0 ? d / 8 : -((7 - d) / 8); }

template <int RS>
struct PlaneBuf {
    static constexpr unsigned ROW = RS * 4, SIZE = RS * ROW;   // bytes
};

extern __shared__ __align__(1024) unsigned char fsm[];

__device__ __forceinline__ float4& word(unsigned off) { return *reinterpret_cast<float4*>(fsm + off); }
__device__ __forceinline__ float2& half_word(unsigned off) { return *reinterpret_cast<float2*>(fsm + off); }

// LP neighbouring values (2 or 4) of a row, as pairs
template <int LP>
__device__ __forceinline__ void load_lines(unsigned off, float2 (&v)[LP / 2]) {
    if constexpr (LP == 4) {
        const float4 q = word(off);
        v[0] = make_float2(q.x, q.y);
        v[1] = make_float2(q.z, q.w);
    } else {
        v[0] = half_word(off);
    }
}
// byte offset of lines LP u .. in a row of the block of eight rows q, row 0 of the block
template <int LP>
__device__ __forceinline__ unsigned line_off(int u, int q) {
    if constexpr (LP == 4) return (unsigned)(u ^ (q & 3)) << 4;
    else return ((unsigned)((u >> 1) ^ (q & 3)) << 4) + ((u & 1) << 3);
}
// NO outputs from NO kb on (along the rows of the buffer at buf, periodic with 8 nb) of the
// lines LP u ..:  acc[k] = sum_t f[k & 1][t] row(NO kb + k - HL + off(k & 1) + t)
// td: the taps, each twice
template <int KIND, int RS, int LP, int NO = 16>
__device__ __forceinline__ void line_item(unsigned buf, int kb, int nb, int u, const float2 (&td)[2][32],
                                          float2 (&acc)[NO][LP / 2]) {
    constexpr int NT = KT<KIND>::NT, HL = KT<KIND>::HL, W = NO + NT - 1 + KT<KIND>::EXTRA;
    constexpr unsigned ROW = PlaneBuf<RS>::ROW;
    constexpr int B0 = floor8(-HL), NB = floor8(W - 1 - HL) - B0 + 1;
    unsigned T[NB];   // the lines' values in the first row of the window's blocks of eight
    #pragma unroll
    for (int b = 0; b < NB; ++b) {
        int q = NO / 8 * kb + B0 + b;
        q += q < 0 ? nb : 0;
        q -= q >= nb ? nb : 0;
        T[b] = buf + q * 8 * ROW + line_off<LP>(u, q);
    }
    #pragma unroll
    for (int k = 0; k < NO; ++k)
        #pragma unroll
        for (int m = 0; m < LP / 2; ++m) acc[k][m] = make_float2(0.f, 0.f);
    static_for<W>([&](auto jc) {
        constexpr int j = decltype(jc)::value, d = j - HL, i = d - 8 * floor8(d);
        float2 v[LP / 2];
        load_lines<LP>((T[floor8(d) - B0] ^ (i << 4)) + i * ROW, v);
        static_for<NO>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            constexpr int t = j - k - ((k & 1) ? KT<KIND>::OFF1 : KT<KIND>::OFF0);
            // (the other filters' parities are equal)
            constexpr int e = KIND == K_SYN || KIND == K_ANA ? k & 1 : 0;
            if constexpr (tap_on<KIND>(t)) {
                #pragma unroll
                for (int m = 0; m < LP / 2; ++m) acc[k][m] = __ffma2_rn(td[e][t], v[m], acc[k][m]);
            }
        });
    });
}
// the item's outputs, transposed: line 2 u + e becomes a row, its words 4 kb + h
template <int RS>
__device__ __forceinline__ unsigned trans_base(unsigned buf, int kb, int u) {
    const int s = (2 * (u & 3)) ^ ((u >> 2) & 3);
    return buf + 2 * u * PlaneBuf<RS>::ROW + ((unsigned)((4 * kb) ^ s) << 4);
}
template <int RS>
__device__ __forceinline__ float4& trans_word(unsigned base, int e, int h) {
    return word((base ^ ((e ^ h) << 4)) + e * PlaneBuf<RS>::ROW);
}
// outputs 4 h .. 4 h + 3 of line e
__device__ __forceinline__ float4 line_word(const float2 (&acc)[16][1], int e, int h) {
    float q[4];
    #pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = e ? acc[4 * h + k][0].y : acc[4 * h + k][0].x;
    return make_float4(q[0], q[1], q[2], q[3]);
}
template <int RS>
__device__ __forceinline__ void store_trans(unsigned buf, int kb, int u, const float2 (&acc)[16][1]) {
    const unsigned base = trans_base<RS>(buf, kb, u);
    #pragma unroll
    for (int e = 0; e < 2; ++e)
        #pragma unroll
        for (int h = 0; h < 4; ++h) trans_word<RS>(base, e, h) = line_word(acc, e, h);
}
// the item's outputs to the global plane of N columns at g
__device__ __forceinline__ void store_global(float* g, int N, int kb, int u, const float2 (&acc)[16][1]) {
    g += (long long)(16 * kb) * N + 2 * u;
    #pragma unroll
    for (int k = 0; k < 16; ++k) *reinterpret_cast<float2*>(g + (long long)k * N) = acc[k][0];
}
// word i (0 to 3) of chunk a (16 columns) of row: (chunk_base(row, a) ^ (i << 4))
template <int RS>
__device__ __forceinline__ unsigned chunk_base(unsigned buf, int row, int a) {
    const unsigned s = swz(row);
    return buf + row * PlaneBuf<RS>::ROW + ((unsigned)(a ^ (int)(s >> 2)) << 6) + ((s & 3) << 4);
}

// Row `row` (periodic with 16 nch columns) from HLR columns before chunk ch on: the window of
// the chunk's outputs
template <int KIND>
struct RowWin {
    static constexpr int HLR = (KT<KIND>::HL + 3) / 4 * 4, D = HLR - KT<KIND>::HL;
    static constexpr int WV = (16 + KT<KIND>::NT - 1 + KT<KIND>::EXTRA + D + 3) / 4;
};
template <int KIND, int RS>
__device__ __forceinline__ void row_win(unsigned buf, int row, int ch, int nch, float (&win)[4 * RowWin<KIND>::WV]) {
    constexpr int HU = RowWin<KIND>::HLR / 4, G = (HU + 3) / 4, PH = 4 * G - HU;
    constexpr int WV = RowWin<KIND>::WV, NG = (PH + WV + 3) / 4;
    unsigned T[NG];
    #pragma unroll
    for (int g = 0; g < NG; ++g) {
        int a = ch - G + g;
        a += a < 0 ? nch : 0;
        a -= a >= nch ? nch : 0;
        T[g] = chunk_base<RS>(buf, row, a);
    }
    static_for<WV>([&](auto qc) {
        constexpr int q = decltype(qc)::value + PH, w = 4 * decltype(qc)::value;
        const float4 v = word(T[q / 4] ^ ((q % 4) << 4));
        win[w] = v.x;
        win[w + 1] = v.y;
        win[w + 2] = v.z;
        win[w + 3] = v.w;
    });
}
// the chunk's outputs; D: the filter's first window element
template <int KIND, int D, int NW>
__device__ __forceinline__ void row_fir(const float (&win)[NW], const float2 (&tp)[32], float (&acc)[16]) {
    #pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0.f;
    const float none[2][32] = {};   // (scalar taps: not used in FP32)
    fir<float, KIND, 16, D>(win, none, tp, acc);
}
template <int RS>
__device__ __forceinline__ void store_chunk(unsigned buf, int row, int ch, const float (&v)[16]) {
    const unsigned b = chunk_base<RS>(buf, row, ch);
    #pragma unroll
    for (int q = 0; q < 4; ++q) word(b ^ (q << 4)) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

// a job: one fine-grid plane (RS x RS) of an orbital
struct Plane {
    const FzSeg<float>* S;
    int I3, o;
    long long base;   // of the plane in the fine arrays
};
__device__ __forceinline__ Plane plane_of(const FzTileParams& p, long long job) {
    int si = 0;
    #pragma unroll 1
    while (si + 1 < p.nseg && job >= p.seg[si + 1].blk0) ++si;
    Plane q;
    q.S = &p.seg[si];
    const long long loc = job - q.S->blk0;
    q.I3 = (int)(loc % q.S->N3);
    q.o = (int)(loc / q.S->N3);
    q.base = (long long)q.o * q.S->P + (long long)q.I3 * q.S->N1 * q.S->N2;
    return q;
}
// starts the copy of the plane at src -> buf as [I2][I1]
template <int RS>
__device__ __forceinline__ void fetch_plane(unsigned buf, const float* src) {
    const int lane = threadIdx.x & 31, nw = (int)(blockDim.x >> 5);
    #pragma unroll 1
    for (int r = threadIdx.x >> 5; r < RS; r += nw) {
        const unsigned s = swz(r);
        for (int u = lane; u < RS / 4; u += 32)
            cp_async16(&word(buf + r * PlaneBuf<RS>::ROW + ((u ^ s) << 4)), src + r * RS + 4 * u);
    }
}

// Items i, i + step, ... of an na x nb grid (b fastest), without a division per item
struct Walk {
    int a, b, da, db, na, nb;
    __device__ __forceinline__ Walk(int i, int step, int na_, int nb_)
        : a(i / nb_), b(i - a * nb_), da(step / nb_), db(step - da * nb_), na(na_), nb(nb_) {}
    template <typename F>
    __device__ __forceinline__ void each(F&& f) const {
        int x = a, y = b;
        #pragma unroll 1
        while (x < na) {
            f(x, y);
            x += da;
            y += db;
            if (y >= nb) {
                y -= nb;
                ++x;
            }
        }
    }
};

template <int PROG, int RS, int REGS>
__global__ void __maxnreg__(REGS) fz_tplane_kernel(const __grid_constant__ FzTileParams p) {
    __shared__ double red[FZ_PTHREADS / 32];
    unsigned X = 0, Z = 2 * PlaneBuf<RS>::SIZE;
    constexpr unsigned Y = PlaneBuf<RS>::SIZE;
    constexpr int N1 = RS, N2 = RS;
    const int T = (int)blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = T >> 5;

    Plane c = plane_of(p, blockIdx.x);
    fetch_plane<RS>(X, c.S->in + c.base);
    cp_commit();
    if (PROG == FZ_MFTA12) {
        fetch_plane<RS>(Z, c.S->in2 + c.base);
        cp_commit();
    }
    #pragma unroll 1
    for (long long job = blockIdx.x; job < p.njobs; job += gridDim.x) {
        const FzSeg<float>& S = *c.S;
        // items along axis 2 ([I2][I1] planes) and along axis 1 ([I1][I2])
        const int nb2 = N2 / 8, nb1 = N1 / 8;
        const Walk w2(threadIdx.x, T, N2 / 16, N1 / 2), w1(threadIdx.x, T, N1 / 16, N2 / 2);
        const bool more = job + gridDim.x < p.njobs;
        Plane nx = c;
        if (more) nx = plane_of(p, job + gridDim.x);
        float2 acc[16][1];

        if constexpr (PROG == FZ_SKM12) {
            cp_wait<0>();
            __syncthreads();   // the plane is here, and the last one is done with
            if (more) {
                fetch_plane<RS>(Z, nx.S->in + nx.base);
                cp_commit();
            }
            // s = S_1 S_2 a -> X
            w2.each([&](int kb, int u) {
                line_item<K_SYN, RS, 2>(X, kb, nb2, u, p.td[0], acc);
                store_trans<RS>(Y, kb, u, acc);
            });
            __syncthreads();
            w1.each([&](int kb, int u) {
                line_item<K_SYN, RS, 2>(Y, kb, nb1, u, p.td[0], acc);
                store_trans<RS>(X, kb, u, acc);
            });
            __syncthreads();
            // eight rows of four columns, as in the general form: the same chains of Ekin
            const Walk we(threadIdx.x, T, N2 / 8, N1 / 4);
            EAcc<float> e;
            // t = MF_2 (MF_1 s in Y), out
            auto put_t = [&](int kb, int u) {
                float2 m[8][2];
                line_item<K_MF, RS, 4, 8>(Y, kb, nb2, u, p.td[3], m);
                float* const g = S.out3 + c.base + (long long)(8 * kb) * N1 + 4 * u;
                #pragma unroll
                for (int k = 0; k < 8; ++k)
                    *reinterpret_cast<float4*>(g + (long long)k * N1) = make_float4(m[k][0].x, m[k][0].y, m[k][1].x, m[k][1].y);
            };
            // v = T_2 s + T_1 s, out if asked for, and its part <s, v>; t1(k): T_1 s at row k
            auto put_v = [&](int kb, int u, auto&& t1) {
                float2 m[8][2];
                line_item<K_KIN, RS, 4, 8>(X, kb, nb2, u, p.td[2], m);
                const unsigned o = X + kb * 8 * PlaneBuf<RS>::ROW + line_off<4>(u, kb);
                float ei = 0.f;
                #pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float4 s = word((o ^ (k << 4)) + k * PlaneBuf<RS>::ROW), a = t1(k);
                    const float4 v = make_float4(m[k][0].x + a.x, m[k][0].y + a.y, m[k][1].x + a.z, m[k][1].y + a.w);
                    ei = fmaf(s.x, v.x, ei);
                    ei = fmaf(s.y, v.y, ei);
                    ei = fmaf(s.z, v.z, ei);
                    ei = fmaf(s.w, v.w, ei);
                    if (S.out2 != nullptr)
                        *reinterpret_cast<float4*>(S.out2 + c.base + (long long)(8 * kb + k) * N1 + 4 * u) = v;
                }
                e.add(ei);
            };
            const int nch = N1 / 16;
            const Walk wr(warp, nw, nch, N2 / 32);   // chunks of 16 columns, blocks of 32 rows
            if (S.part != nullptr && S.out2 != nullptr) {
                // H psi: T_1 s -> v and MF_1 s -> Y from one window
                wr.each([&](int ch, int rb) {
                    const int row = rb * 32 + lane;
                    float win[4 * RowWin<K_KIN>::WV], v[16];
                    row_win<K_KIN, RS>(X, row, ch, nch, win);
                    row_fir<K_KIN, RowWin<K_KIN>::D>(win, p.tp[0], v);
                    if constexpr (RS == 128) {
                        // through the item's own place in Y, so that four lanes write 64 bytes
                        // of a row: 128^2 746 against 797, 96^2 425 against 414
                        store_chunk<RS>(Y, row, ch, v);
                        __syncwarp();
                        #pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int r = rb * 32 + 8 * i + ((lane >> 2 & 1) << 2) + (lane >> 3), q = lane & 3;
                            *reinterpret_cast<float4*>(S.out2 + c.base + (long long)r * N1 + 16 * ch + 4 * q) =
                                word(chunk_base<RS>(Y, r, ch) ^ (q << 4));
                        }
                        __syncwarp();
                    } else {
                        float4* const g = reinterpret_cast<float4*>(S.out2 + c.base + (long long)row * N1 + 16 * ch);
                        #pragma unroll
                        for (int q = 0; q < 4; ++q)
                            g[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                    }
                    row_fir<K_MF, RowWin<K_KIN>::HLR - KT<K_MF>::HL>(win, p.tp[1], v);
                    store_chunk<RS>(Y, row, ch, v);
                });
                __syncthreads();
                we.each([&](int kb, int u) {
                    put_t(kb, u);
                    const float* const g = S.out2 + c.base + (long long)(8 * kb) * N1 + 4 * u;
                    float4 t1[8];
                    #pragma unroll
                    for (int k = 0; k < 8; ++k) t1[k] = *reinterpret_cast<const float4*>(g + (long long)k * N1);
                    put_v(kb, u, [&](int k) { return t1[k]; });
                });
            } else {
                if (S.part != nullptr) {
                    wr.each([&](int ch, int rb) {
                        const int row = rb * 32 + lane;
                        float win[4 * RowWin<K_KIN>::WV], v[16];
                        row_win<K_KIN, RS>(X, row, ch, nch, win);
                        row_fir<K_KIN, RowWin<K_KIN>::D>(win, p.tp[0], v);
                        store_chunk<RS>(Y, row, ch, v);
                    });
                    __syncthreads();
                    we.each([&](int kb, int u) {
                        const unsigned o = Y + kb * 8 * PlaneBuf<RS>::ROW + line_off<4>(u, kb);
                        put_v(kb, u, [&](int k) { return word((o ^ (k << 4)) + k * PlaneBuf<RS>::ROW); });
                    });
                    __syncthreads();
                }
                wr.each([&](int ch, int rb) {
                    const int row = rb * 32 + lane;
                    float win[4 * RowWin<K_MF>::WV], v[16];
                    row_win<K_MF, RS>(X, row, ch, nch, win);
                    row_fir<K_MF, RowWin<K_MF>::D>(win, p.tp[1], v);
                    store_chunk<RS>(Y, row, ch, v);
                });
                __syncthreads();
                we.each([&](int kb, int u) { put_t(kb, u); });
            }
            if (S.part != nullptr) {
                const double tot = fz_block_sum(e, red);
                if (threadIdx.x == 0) S.part[(long long)c.o * S.ptiles + S.poff + c.I3] = tot;
            }
        } else {
            cp_wait<1>();      // x; v may still be under way
            __syncthreads();
            // w = MFT_2 MFT_1 x + v -> X, MFT_1 first as in the general form
            const int nch = N1 / 16;
            const Walk wr(warp, nw, nch, N2 / 32);   // a lane per I2, chunks of 16
            wr.each([&](int ch, int rb) {
                const int row = rb * 32 + lane;
                float win[4 * RowWin<K_MFT>::WV], v[16];
                row_win<K_MFT, RS>(X, row, ch, nch, win);
                row_fir<K_MFT, RowWin<K_MFT>::D>(win, p.tp[1], v);
                store_chunk<RS>(Y, row, ch, v);
            });
            cp_wait<0>();
            __syncthreads();
            w2.each([&](int kb, int u) {
                line_item<K_MFT, RS, 2>(Y, kb, nb2, u, p.td[0], acc);
                #pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const unsigned o = (2 * kb + h) * 8 * PlaneBuf<RS>::ROW + line_off<2>(u, 2 * kb + h);
                    #pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float2 v = half_word(((Z + o) ^ (k << 4)) + k * PlaneBuf<RS>::ROW);
                        half_word(((X + o) ^ (k << 4)) + k * PlaneBuf<RS>::ROW) =
                            make_float2(acc[8 * h + k][0].x + v.x, acc[8 * h + k][0].y + v.y);
                    }
                }
            });
            __syncthreads();
            if (more) fetch_plane<RS>(Z, nx.S->in + nx.base);
            cp_commit();
            // w' = A_2 A_1 w
            wr.each([&](int ch, int rb) {
                const int row = rb * 32 + lane;
                float win[4 * RowWin<K_ANA>::WV], v[16];
                row_win<K_ANA, RS>(X, row, ch, nch, win);
                row_fir<K_ANA, RowWin<K_ANA>::D>(win, p.tp[0], v);
                store_chunk<RS>(Y, row, ch, v);
            });
            __syncthreads();
            if (more) fetch_plane<RS>(X, nx.S->in2 + nx.base);
            cp_commit();
            w2.each([&](int kb, int u) {
                line_item<K_ANA, RS, 2>(Y, kb, nb2, u, p.td[1], acc);
                store_global(S.out + c.base, N1, kb, u, acc);
            });
        }
        c = nx;
        const unsigned t = X;
        X = Z;
        Z = t;
    }
}

size_t tplane_smem(FzShape s) { return (s.ctas > 0 ? 3 : 2) * (size_t)s.rs * s.rs * sizeof(float); }

template <typename F>
cudaError_t tplane_pick(int prog, FzShape s, F&& f) {
    if (prog == FZ_SKM12) switch (s.rs) {
        case 128: return f(fz_tplane_kernel<FZ_SKM12, 128, 128>);
        case 96: return f(fz_tplane_kernel<FZ_SKM12, 96, 128>);
        case 64: return f(fz_tplane_kernel<FZ_SKM12, 64, 128>);
        case 32: return f(fz_tplane_kernel<FZ_SKM12, 32, 128>);
        }
    if (prog == FZ_MFTA12) switch (s.rs) {
        case 128: return f(fz_tplane_kernel<FZ_MFTA12, 128, 128>);
        case 96: return f(fz_tplane_kernel<FZ_MFTA12, 96, 96>);
        case 64: return f(fz_tplane_kernel<FZ_MFTA12, 64, 96>);
        }
    return cudaErrorInvalidConfiguration;
}

}  // namespace

// FZ_MFTA12, whose v is a second plane to wait for, always fetches ahead: CTAs that share an SM
// walk over the planes.  FZ_SKM12 does where a plane is alone on its SM; three 96^2 planes
// without a third buffer take 388 where two with one take 444.
FzShape fz_tplane_shape(int prog, int N1, int N2) {
    if (N1 != N2) return {};
    const bool w = prog == FZ_MFTA12;
    switch (N1) {
    case 128: return {512, 128, 128, 1};
    case 96: return w ? FzShape{256, 96, 96, 2} : FzShape{160, 128, 96, 0};
    case 64: return w ? FzShape{128, 96, 64, 4} : FzShape{64, 128, 64, 0};
    case 32: return w ? FzShape{} : FzShape{32, 128, 32, 0};
    }
    return {};
}

cudaError_t prepare_tplane(int prog, FzShape s) {
    // large dynamic shared memory once per device and kernel
    static std::atomic<unsigned long long> done[2][5];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    std::atomic<unsigned long long>& d = done[prog == FZ_SKM12][s.rs / 32];
    if (d.load() & bit) return cudaSuccess;
    e = tplane_pick(prog, s, [&](auto* k) {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tplane_smem(s));
    });
    if (e == cudaSuccess) d.fetch_or(bit);
    return e;
}

cudaError_t launch_tplane(int prog, const FzParams<float>& p, cudaStream_t st) {
    FzTileParams q;
    const int nk = prog == FZ_SKM12 ? 4 : 2;
    for (int m = 0; m < nk; ++m)
        for (int e = 0; e < 2; ++e)
            for (int t = 0; t < 32; ++t) q.td[m][e][t] = make_float2(p.tap[m][e][t], p.tap[m][e][t]);
    if (prog == FZ_SKM12) {
        tap_pairs<K_KIN>(p.tap[1], q.tp[0]);
        tap_pairs<K_MF>(p.tap[3], q.tp[1]);
    } else {
        tap_pairs<K_ANA>(p.tap[1], q.tp[0]);
        tap_pairs<K_MFT>(p.tap[0], q.tp[1]);
    }
    q.njobs = p.njobs;
    q.nseg = p.nseg;
    for (int k = 0; k < p.nseg; ++k) q.seg[k] = p.seg[k];
    cudaError_t e = prepare_tplane(prog, p.shape);
    if (e != cudaSuccess) return e;
    return tplane_pick(prog, p.shape, [&](auto* k) {
        long long grid = p.njobs;
        if (p.shape.ctas > 0) {
            int dev = 0, nsm = 0;
            cudaError_t r = cudaGetDevice(&dev);
            if (r == cudaSuccess) r = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
            if (r != cudaSuccess) return r;
            grid = std::min(grid, (long long)nsm * p.shape.ctas);
        }
        k<<<dim3((unsigned)grid), dim3(p.shape.threads), tplane_smem(p.shape), st>>>(q);
        count_launches(1);
        return cudaGetLastError();
    });
}

}  // namespace wvl
