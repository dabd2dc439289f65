// Orbital scalar products on the FP16 tensor cores:
//   S[i][j] = sum_k a_i[k] b_j[k]   (Sec. "Daubechies basis and wavelet
// transformation": the compressed basis is orthonormal)
// as a dense contraction of exact integer digits.
//
// Every row's part in a slice of k is put on its own power-of-two scale (its largest
// exponent, from a first read) and rounded to an integer |X| < 2^55,
// which seven signed base-256 digits hold: X = sum_q x_q 256^(6 - q),
// |x_q| <= 128, exact in FP16.  The products of digit q of a_i and digit p of
// b_j have weight 256^(12 - q - p); the pairs of one diagonal s = q + p share
// an FP32 accumulator.  A digit product is at most 2^14 and a diagonal has at
// most 7 of them per k, so over OM_KC = 128 coefficients every partial sum is
// an integer below 7 * 128 * 2^14 < 2^24: exact in any order.  The
// accumulators are then added into two 64-bit integers per entry
// (diagonals 0..2 and 3..6).  The only roundings are those of the inputs (2^-56 of
// the slice's largest magnitude, none for FP32 inputs down to 2^-32 of it), the
// dropped diagonals s >= 7 (below 2^-53 of one product of the largest magnitudes,
// of random sign) and one FP64 addition per slice -- no rounding per term, which an
// FP64 sum of len terms has.
// Rows with an infinity or a NaN have no scale: their entries are summed in
// FP64 by the reduction.
//
// Bound: the FP64 FMA loop this replaces runs on a pipe of 1.7 lanes per clock and SM.
// Here a CTA (one per SM) owns 128 x 64 entries and a slice of k and walks it in
// stages of 32 k: 12 warps slice into the digit planes (K-major core matrices, two
// stages in shared memory) while the MMAs of the stage before, issued by one
// thread of another warp, run: per 16 k, digit q of a against digits 0 .. 6 - q of b
// side by side along N, 28 pairs in 10 instructions.  All 16 warps read the
// accumulators.  256 FP32 vectors of 884736 coefficients, symmetric: 72.4 -> 2.6 ms (the
// FP64 loop's error of 4.4e-14, relative to the whole matrix, becomes 2.1e-15);
// 4 vectors: 1640 -> 360 us; 64 x 64 of 64 coefficients: both at the launches'
// 26 us.  The MMAs issued by one of the slicing warps measured 4.1 ms (an issue
// blocks while the queue is full, and the warp's stage waits for it).  What is left:
// the tensor cores are busy for about 45 % of the time, the rest is the slicing of a
// stage (the warps' issue slots) and the reading of the accumulators, during which
// they idle.
#include <algorithm>
#include <cstdint>

#include <cuda_fp16.h>

#include "tcgen05.cuh"
#include "wvl.h"
#include "wvl_internal.h"

namespace wvl {

__device__ unsigned int g_om_timeouts = 0;

namespace {

using namespace tc;

constexpr int OM_M = 128, OM_N = 64;      // entries per CTA
constexpr int OM_D = 7;                   // digits
constexpr int OM_KS = 32;                 // k per stage
constexpr int OM_KC = 128;                // k per accumulation in tensor memory
constexpr int OM_THREADS = 512;
constexpr int OM_SLICE = 12;              // slicing warps; the next one issues the MMAs
constexpr int OM_CH = OM_KS / 8;          // 8-k chunks per stage
// chunk strides (the MMA's leading-dimension offset), with 64 bytes of skew: the
// eight lanes of a store phase hold two chunks x four rows
constexpr int OM_LBOA = OM_M * 16 + 64, OM_LBOB = OM_D * OM_N * 16 + 64;
constexpr int OM_APL = OM_CH * OM_LBOA;   // digit plane of a
constexpr int OM_ABYTES = OM_D * OM_APL, OM_STAGE = OM_ABYTES + OM_CH * OM_LBOB;
constexpr int OM_SMEM = 2 * OM_STAGE;
constexpr int OM_SLOTS = 152;             // CTAs resident at once (one per SM)
static_assert(7LL * OM_KC * (1 << 14) < (1 << 24), "exact partial sums");

struct OmParams {
    const void* a;
    const void* b;
    longlong2* part;     // [nsplit][na][nb]: diagonals 0..2 and 3..6
    const int* rexp;     // [rows][nsplit] largest biased exponents: rows of a, then of b
    long long len, kper;
    int na, nb, nsplit, tiles_j, sym;
    int brow;            // first row of b in rexp (0 when a is b)
};

template <typename T> struct Bits;
template <> struct Bits<float> {
    static constexpr int EMAX = 255, BIAS = 181;      // x = X 2^(E - BIAS)
    __device__ static int expo(float x) { return (int)((__float_as_uint(x) >> 23) & 255u); }
};
template <> struct Bits<double> {
    static constexpr int EMAX = 2047, BIAS = 1077;
    __device__ static int expo(double x) { return (int)((__double2hiint(x) >> 20) & 2047); }
};

// X + 0x80808080808080 for X = round(x 2^(BIAS - E)), E the row's largest
// biased exponent (subnormals count as exponent 1 without the hidden bit)
__device__ __forceinline__ unsigned long long biased(unsigned long long m2, int d, bool neg) {
    d = d > 63 ? 63 : d;
    const unsigned long long r = ((m2 >> d) + 1) >> 1;
    constexpr unsigned long long C = 0x80808080808080ULL;
    return neg ? C - r : C + r;
}
__device__ __forceinline__ unsigned long long biased(double x, int E) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((u >> 52) & 2047u);
    const unsigned long long m = (u & ((1ULL << 52) - 1)) | (e ? 1ULL << 52 : 0ULL);
    return biased(m << 3, E - max(e, 1), (long long)u < 0);
}

// NV (8 or 4) consecutive elements from k (a multiple of NV) of a row, zero from k1 on
template <typename T, int NV>
__device__ __forceinline__ void load_k(const T* __restrict__ row, long long k, long long k1, bool vec,
                                       T (&v)[NV]) {
    constexpr int PER = 16 / (int)sizeof(T);
    if (vec && k + NV <= k1) {
        #pragma unroll
        for (int q = 0; q < NV / PER; ++q) {
            if constexpr (sizeof(T) == 4) {
                const float4 f = __ldg(reinterpret_cast<const float4*>(row + k) + q);
                v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
            } else {
                const double2 f = __ldg(reinterpret_cast<const double2*>(row + k) + q);
                v[2 * q] = f.x; v[2 * q + 1] = f.y;
            }
        }
        return;
    }
    #pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = k + q < k1 ? row[k + q] : T(0);
}

// the FP16 patterns 0x6480 + digit (the values 1152 + digit) of a plane's pairs ->
// the digits, stored as one 16- or 8-byte word
template <int NP>
__device__ __forceinline__ void put_digits(unsigned char* dst, const unsigned (&p)[NP]) {
    const __half2 off = __halves2half2(__ushort_as_half((unsigned short)0x6480),
                                       __ushort_as_half((unsigned short)0x6480));
    unsigned w[NP];
    #pragma unroll
    for (int i = 0; i < NP; ++i) {
        const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&p[i]), off);
        w[i] = *reinterpret_cast<const unsigned*>(&h);
    }
    if constexpr (NP == 4) *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    else *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
}

// The digits of NV elements, one word per digit plane (stride pl).
// FP32: with |y| < 128, y = x 2^(133 - E), digit q is y rounded to a multiple of
// 2^(-8 q), taken off y exactly before the next one (digits in [-128, 128]); adding
// 12608640 2^(-8 q) rounds, and leaves 0x6480 + digit in the low half of the
// sum's bits.  Packed additions on the FMA pipe: the integer form (below,
// for FP64) kept the ALU pipe 37 % busy and was 1.9 times slower.
template <int NV>
__device__ __forceinline__ void store_digits(unsigned char* dst, int pl, const float (&v)[NV], float2 s0,
                                             float2 s1) {
    const float2 m1 = make_float2(-1.f, -1.f);
    float2 y[NV / 2];
    #pragma unroll
    for (int i = 0; i < NV / 2; ++i)
        y[i] = __fmul2_rn(__fmul2_rn(make_float2(v[2 * i], v[2 * i + 1]), s0), s1);
    float m = 12608640.f;
    #pragma unroll
    for (int q = 0; q < OM_D; ++q, m *= 1.f / 256.f) {
        unsigned p[NV / 2];
        #pragma unroll
        for (int i = 0; i < NV / 2; ++i) {
            const float2 t = __fadd2_rn(y[i], make_float2(m, m));
            const float2 d = __fadd2_rn(t, make_float2(-m, -m));
            y[i] = __ffma2_rn(d, m1, y[i]);
            p[i] = __byte_perm(__float_as_uint(t.x), __float_as_uint(t.y), 0x5410);
        }
        put_digits<NV / 2>(dst + q * pl, p);
    }
}
__device__ __forceinline__ float pow2(int e) { return __int_as_float((e + 127) << 23); }
template <int NV>
__device__ __forceinline__ void store_digits(unsigned char* dst, int pl, const float (&v)[NV], int E) {
    const int e = 133 - E, h = e >> 1;   // in two factors: 2^132 is no float
    const float a = pow2(h), b = pow2(e - h);
    store_digits<NV>(dst, pl, v, make_float2(a, a), make_float2(b, b));
}
// FP64: the bytes of X + 128 sum_q 256^q are the digits 6 .. 1 plus 128 (digits in
// [-128, 127]), its top half word is digit 0 plus 128
template <int NV>
__device__ __forceinline__ void store_digits(unsigned char* dst, int pl, const double (&v)[NV], int E) {
    unsigned lo[NV], hi[NV];
    #pragma unroll
    for (int q = 0; q < NV; ++q) {
        const unsigned long long y = biased(v[q], E);
        lo[q] = (unsigned)y;
        hi[q] = (unsigned)(y >> 32);
    }
    constexpr unsigned H = 0x64646464u;
    unsigned p[NV / 2], g[NV / 2];
    #pragma unroll
    for (int i = 0; i < NV / 2; ++i) p[i] = __byte_perm(hi[2 * i], hi[2 * i + 1], 0x7632) + 0x64006400u;
    put_digits<NV / 2>(dst, p);
    #pragma unroll
    for (int w = 0; w < 3; ++w) {   // digits 1, 2 from the high word, 3 .. 6 from the low one
        #pragma unroll
        for (int i = 0; i < NV / 2; ++i)
            g[i] = w == 0 ? __byte_perm(hi[2 * i], hi[2 * i + 1], 0x5410)
                          : __byte_perm(lo[2 * i], lo[2 * i + 1], w == 1 ? 0x7632 : 0x5410);
        #pragma unroll
        for (int i = 0; i < NV / 2; ++i) p[i] = __byte_perm(g[i], H, 0x4341);
        put_digits<NV / 2>(dst + (2 * w + 1) * pl, p);
        #pragma unroll
        for (int i = 0; i < NV / 2; ++i) p[i] = __byte_perm(g[i], H, 0x4240);
        put_digits<NV / 2>(dst + (2 * w + 2) * pl, p);
    }
}

// largest biased exponent of a row's slice, at least 1 (the scale of subnormals)
__device__ __forceinline__ int row_exp(const OmParams& q, int row, int split) {
    return max(1, q.rexp[(long long)row * q.nsplit + split]);
}

// one block per (slice, row)
template <typename T>
__global__ void __launch_bounds__(256) row_exp_kernel(const OmParams q, int row0, int* __restrict__ rexp) {
    __shared__ int red[8];
    const int r = row0 + blockIdx.y;
    const T* x = r < q.na ? static_cast<const T*>(q.a) + (long long)r * q.len
                          : static_cast<const T*>(q.b) + (long long)(r - q.na) * q.len;
    constexpr int PER = 16 / (int)sizeof(T);
    const long long k0 = (long long)blockIdx.x * q.kper, k1 = min(q.len, k0 + q.kper);
    int e = 0;
    if (q.len % PER == 0) {
        #pragma unroll 4
        for (long long k = k0 + threadIdx.x * PER; k < k1; k += 256 * PER) {
            if constexpr (sizeof(T) == 4) {
                const float4 f = __ldg(reinterpret_cast<const float4*>(x + k));
                e = max(max(e, max(Bits<T>::expo(f.x), Bits<T>::expo(f.y))),
                        max(Bits<T>::expo(f.z), Bits<T>::expo(f.w)));
            } else {
                const double2 f = __ldg(reinterpret_cast<const double2*>(x + k));
                e = max(e, max(Bits<T>::expo(f.x), Bits<T>::expo(f.y)));
            }
        }
    } else {
        #pragma unroll 4
        for (long long k = k0 + threadIdx.x; k < k1; k += 256) e = max(e, Bits<T>::expo(x[k]));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) e = max(e, red[w]);
        rexp[(long long)r * q.nsplit + blockIdx.x] = e;
    }
}

template <typename T>
__global__ void __launch_bounds__(OM_THREADS, 1) overlap_mma_kernel(const OmParams q) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ uint32_t tslot;
    __shared__ __align__(8) uint64_t full[2], empty[2], done, drained;
    __shared__ volatile int dead;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // tile (ti, tj); when symmetric only the tiles that reach the diagonal or
    // lie above it, tj >= 2 ti
    int ti, tj;
    if (q.sym) {
        int r = blockIdx.y, t = 0;
        while (r >= q.tiles_j - 2 * t) { r -= q.tiles_j - 2 * t; ++t; }
        ti = t;
        tj = 2 * t + r;
    } else {
        ti = blockIdx.y / q.tiles_j;
        tj = blockIdx.y - ti * q.tiles_j;
    }
    const int i0 = ti * OM_M, j0 = tj * OM_N;
    const long long k0 = (long long)blockIdx.x * q.kper;
    const long long k1 = min(q.len, k0 + q.kper);
    const int nst = (int)((k1 - k0 + OM_KS - 1) / OM_KS);
    const bool vec = q.len % (16 / (int)sizeof(T)) == 0;

    // a slicing thread's share of a stage: 8 k (chunk ch) of two rows of the tile's 192
    // (128 of a, then 64 of b); a warp covers 8 rows x 32 k at a time, and the
    // lanes of a store phase fall on distinct banks
    const int ch = (lane & 1) | ((lane >> 2) & 2);
    const T* row[2] = {nullptr, nullptr};
    int dst[2], pl[2], E[2];
    #pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int r = (warp + u * OM_SLICE) * 8 + (((lane >> 1) & 3) | ((lane >> 2) & 4));
        const bool isa = r < OM_M;
        const int g = isa ? i0 + r : j0 + r - OM_M;
        const bool on = warp < OM_SLICE && g < (isa ? q.na : q.nb);
        if (on) row[u] = static_cast<const T*>(isa ? q.a : q.b) + (long long)g * q.len;
        dst[u] = isa ? ch * OM_LBOA + r * 16 : OM_ABYTES + ch * OM_LBOB + (r - OM_M) * 16;
        pl[u] = isa ? OM_APL : OM_N * 16;
        E[u] = on ? row_exp(q, isa ? g : q.brow + g, blockIdx.x) : 1;
    }

    // both stages start at zero, which rows past the ends keep
    for (int i = tid * 16; i < OM_SMEM; i += OM_THREADS * 16)
        *reinterpret_cast<uint4*>(sm + i) = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (tid == 0) {
        auto init = [](uint64_t& b, int n) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(su32(&b)), "r"(n));
        };
        init(full[0], OM_SLICE);
        init(full[1], OM_SLICE);
        init(empty[0], 1);
        init(empty[1], 1);
        init(done, 1);
        init(drained, OM_THREADS / 32);
        dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(su32(&tslot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tm = tslot;
    // Stage st is the (st / 2)-th use of its buffer's barriers: full, one arrival per
    // slicing warp once its digits are stored; empty, the commit of the MMAs that read them.
    // Per accumulation: done, the commit of its last MMAs; drained, one arrival per
    // warp once it has read the accumulators.  Whoever waits on a barrier waits for
    // every use of it in turn (a parity tells neighbouring uses apart only).  A
    // wait that runs out ends every other one.
    auto wait = [&](uint64_t& bar, int use) -> bool {
        const uint32_t addr = su32(&bar), parity = (uint32_t)use & 1u;
        const long long t0 = clock64();
        bool got = false;
        while (!got && !dead) {
            uint32_t ok;
            asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                         "selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
            got = ok != 0;
            if (!got && clock64() - t0 > WAIT_CYCLES) dead = 1;
        }
        return __all_sync(0xffffffffu, got);
    };
    auto arrive = [&](uint64_t& bar) {
        __syncwarp();
        if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(su32(&bar)) : "memory");
    };
    constexpr int SPC = OM_KC / OM_KS;   // stages per accumulation

    // entries of this thread: row 32 (warp % 4) + lane, columns 16 (warp / 4) .. + 15
    const int er = 32 * (warp & 3) + lane, ec = 16 * (warp >> 2);
    const uint32_t tl = tm + ((uint32_t)(32 * (warp & 3)) << 16) + ec;
    // their sums hi 2^32 + lo
    long long hi[16];
    unsigned lo[16];
    #pragma unroll
    for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0;

    // the accumulators of the last OM_KC (or fewer) k into the integers: diagonals
    // 3..6 (below 2^48 in units of diagonal 6), whose carry joins diagonals 0..2
    auto drain = [&]() {
        fence_after();
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t v[OM_D][8];
            #pragma unroll
            for (int s = 0; s < OM_D; ++s) tld8(tl + s * OM_N + 8 * h, v[s]);
            tld_wait();
            #pragma unroll
            for (int c = 0; c < 8; ++c) {
                long long t = lo[8 * h + c];
                #pragma unroll
                for (int s = 3; s < OM_D; ++s)
                    t += (long long)__float2int_rn(__uint_as_float(v[s][c])) * (1 << (8 * (6 - s)));
                lo[8 * h + c] = (unsigned)t;
                t >>= 32;
                #pragma unroll
                for (int s = 0; s < 3; ++s)
                    t += (long long)__float2int_rn(__uint_as_float(v[s][c])) * (1 << (8 * (2 - s)));
                hi[8 * h + c] += t;
            }
        }
        fence_before();
        arrive(drained);
    };

    bool ok = true;
    // the accumulation before stage st (or the last one) read by every warp
    auto drain_before = [&](int st) {
        if (st > 0 && (st % SPC == 0 || st == nst))
            if ((ok = wait(done, (st - 1) / SPC))) drain();
    };
    if (warp < OM_SLICE) {
        T v[2][8];
        constexpr bool AHEAD = sizeof(T) == 4;   // the next stage's loads in flight under this one
        auto load = [&](int st) {
            const long long k = k0 + (long long)st * OM_KS + 8 * ch;
            #pragma unroll
            for (int u = 0; u < 2; ++u)
                if (row[u] != nullptr) load_k<T, 8>(row[u], k, k1, vec, v[u]);
        };
        if (AHEAD) load(0);
        #pragma unroll 1
        for (int st = 0; st <= nst && ok; ++st) {
            if (st < nst) {
                if (st >= 2 && !(ok = wait(empty[st & 1], (st >> 1) - 1))) break;
                unsigned char* const A = sm + (st & 1) * OM_STAGE;
                if (!AHEAD) load(st);
                #pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (row[u] != nullptr) store_digits<8>(A + dst[u], pl[u], v[u], E[u]);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                arrive(full[st & 1]);
                if (AHEAD && st + 1 < nst) load(st + 1);
            }
            drain_before(st);
        }
    } else if (warp == OM_SLICE) {
        // one thread issues the MMAs: an issue blocks while the tensor cores' queue is
        // full, so a slicing warp that issued would hold up its stage
        int st = 0;
        for (; st <= nst; ++st) {
            drain_before(st);
            if (!ok || st == nst) break;
            const bool first = st % SPC == 0;
            if (!(ok = wait(full[st & 1], st >> 1))) break;
            if (first && st > 0 && !(ok = wait(drained, st / SPC - 1))) break;
            if (lane == 0) {
                fence_after();
                const unsigned char* const A = sm + (st & 1) * OM_STAGE;
                const uint64_t ad = mdesc(su32(A), OM_LBOA, 128);
                const uint64_t bd = mdesc(su32(A + OM_ABYTES), OM_LBOB, 128);
                #pragma unroll
                for (int ks = 0; ks < OM_KS / 16; ++ks)
                    #pragma unroll
                    for (int dq = 0; dq < OM_D; ++dq)
                        #pragma unroll
                        for (int fp = 0; fp < OM_D - dq; fp += 4) {
                            const int nd = OM_D - dq - fp < 4 ? OM_D - dq - fp : 4;
                            mma(tm + (dq + fp) * OM_N,
                                ad + (uint64_t)((dq * OM_APL + 2 * ks * OM_LBOA) >> 4),
                                bd + (uint64_t)((2 * ks * OM_LBOB + fp * OM_N * 16) >> 4),
                                idesc_f16(OM_M, nd * OM_N), (first && ks == 0 && dq == 0) ? 0u : 1u);
                        }
                commit(su32(&empty[st & 1]));
                if (st % SPC == SPC - 1 || st == nst - 1) commit(su32(&done));
            }
            __syncwarp();
        }
        if (!ok && lane == 0) {
            // let the MMAs in flight finish (bounded) before the accumulators are freed
            const int uses = st / SPC;   // of done so far
            commit(su32(&done));
            if (uses > 0) wait_parity(su32(&done), (uint32_t)(uses - 1) & 1u);
            wait_parity(su32(&done), (uint32_t)uses & 1u);
        }
        __syncwarp();
    } else {
        #pragma unroll 1
        for (int st = SPC; st < nst + SPC && ok; st += SPC) drain_before(min(st, nst));
    }
    if (ok && i0 + er < q.na) {
        longlong2* const P = q.part + ((long long)blockIdx.x * q.na + i0 + er) * q.nb + j0 + ec;
        #pragma unroll
        for (int c = 0; c < 16; ++c)
            if (j0 + ec + c < q.nb) P[c] = make_longlong2(hi[c], (long long)lo[c]);
    }
    fence_before();
    __syncthreads();
    if (tid == 0 && dead) atomicAdd(&g_om_timeouts, 1u);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tm), "r"(512));
}

// S[i][j] = the slices' integers, each scaled, added in a fixed order by rl lanes
// (one lane walking 152 slices is a chain of loads that took 40 us); when symmetric,
// entries of tiles left of the diagonal
// blocks take the mirrored one.  Entries of a row without a scale (infinity or
// NaN) are summed in FP64 by the whole block, one after another.
template <typename T>
__global__ void __launch_bounds__(256) overlap_mma_reduce_kernel(const OmParams q, int rl, double* __restrict__ S) {
    __shared__ int plain[256];
    __shared__ double red[8];
    const long long n = (long long)q.na * q.nb;
    const T* const A = static_cast<const T*>(q.a);
    const T* const B = static_cast<const T*>(q.b);
    const int EB = 256 / rl;   // entries per block and turn
    #pragma unroll 1
    for (long long base = (long long)blockIdx.x * EB; base < n; base += (long long)gridDim.x * EB) {
        const int part = threadIdx.x % rl;
        const long long e = base + threadIdx.x / rl;
        int bad = 0;
        double t = 0.0;
        if (e < n) {
            int i = (int)(e / q.nb), j = (int)(e - (long long)i * q.nb);
            if (q.sym && j / OM_N < 2 * (i / OM_M)) { const int u = i; i = j; j = u; }
            #pragma unroll 4
            for (int s = part; s < q.nsplit; s += rl) {
                const int Ea = row_exp(q, i, s), Eb = row_exp(q, q.brow + j, s);
                const longlong2 v = q.part[(long long)s * n + (long long)i * q.nb + j];
                bad |= Ea == Bits<T>::EMAX || Eb == Bits<T>::EMAX;
                // x 2^32 + y, in units of 2^48 of the integers' product
                t += scalbn(fma((double)v.x, 4294967296.0, (double)v.y), 48 + Ea + Eb - 2 * Bits<T>::BIAS);
            }
        }
        #pragma unroll 1
        for (int off = rl / 2; off > 0; off >>= 1) {
            t += __shfl_down_sync(0xffffffffu, t, off, rl);
            bad |= __shfl_down_sync(0xffffffffu, bad, off, rl);
        }
        if (e < n && part == 0 && !bad) S[e] = t;
        bad &= part == 0;
        if (!__syncthreads_or(bad)) continue;
        if (part == 0) plain[threadIdx.x / rl] = bad;
        __syncthreads();
        #pragma unroll 1
        for (int c = 0; c < EB; ++c) {
            if (!plain[c]) continue;
            const long long ec = base + c;
            const int i = (int)(ec / q.nb), j = (int)(ec - (long long)i * q.nb);
            double s = 0.0;
            for (long long k = threadIdx.x; k < q.len; k += 256)
                s = fma((double)A[(long long)i * q.len + k], (double)B[(long long)j * q.len + k], s);
            #pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
            if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int w = 1; w < 8; ++w) s += red[w];
                S[ec] = s;
            }
            __syncthreads();
        }
    }
}

// Slices of k: whole accumulations of OM_KC, as many as minimise the waves of
// CTAs (one per SM) times a slice's length, each CTA costing about four
// accumulations more (start, exponents, partials).  The same on every GPU, so that the
// workspace bound holds.
void om_shape(int na, int nb, long long len, bool sym, int& nsplit, long long& kper, long long& tiles) {
    const long long ti = (na + OM_M - 1) / OM_M, tj = (nb + OM_N - 1) / OM_N;
    tiles = sym ? ti * tj - ti * (ti - 1) : ti * tj;
    const long long chunks = std::max(1LL, (len + OM_KC - 1) / OM_KC);
    long long best = -1, ns = 1;
    for (long long s = 1; s <= std::min(chunks, 2LL * OM_SLOTS); ++s) {
        const long long cost = (tiles * s + OM_SLOTS - 1) / OM_SLOTS * ((chunks + s - 1) / s + 4);
        if (best < 0 || cost < best) {
            best = cost;
            ns = s;
        }
    }
    // a slice's low integer takes 2^47 per accumulation
    ns = std::max(ns, (chunks + 32767) / 32768);
    kper = (chunks + ns - 1) / ns * OM_KC;
    nsplit = (int)((chunks * OM_KC + kper - 1) / kper);
}

template <typename T>
cudaError_t run_om(const OmParams& q, long long tiles, int* rexp, double* S, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(overlap_mma_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         OM_SMEM);
    if (e != cudaSuccess) return e;
    const int rows = q.na + (q.brow ? q.nb : 0);
    for (int r0 = 0; r0 < rows; r0 += 65535) {   // (the grid's y limit)
        row_exp_kernel<T><<<dim3((unsigned)q.nsplit, (unsigned)std::min(rows - r0, 65535)), 256, 0, st>>>(
            q, r0, rexp);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    overlap_mma_kernel<T><<<dim3((unsigned)q.nsplit, (unsigned)tiles), OM_THREADS, OM_SMEM, st>>>(q);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const long long n = (long long)q.na * q.nb;
    int rl = 1;   // lanes per entry: more only where the entries alone are few
    while (rl < 16 && n * rl < 32768 && q.nsplit >= 8 * rl) rl *= 2;
    const long long blocks = std::min<long long>((n * rl + 255) / 256, 152LL * 8);
    overlap_mma_reduce_kernel<T><<<(unsigned)blocks, 256, 0, st>>>(q, rl, S);
    count_launches(1);
    return cudaGetLastError();
}

size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

}  // namespace

size_t overlap_mma_ws(int na, int nb, long long len, bool sym) {
    int ns = 1;
    long long kper = 0, tiles = 0;
    om_shape(na, nb, len, sym, ns, kper, tiles);
    const size_t rows = (size_t)na + (sym ? 0 : nb);
    return align16(rows * ns * sizeof(int)) + (size_t)ns * na * nb * sizeof(longlong2);
}

cudaError_t launch_overlap_mma(int prec, int na, const void* a, int nb, const void* b, long long len,
                               bool sym, double* S, void* ws, cudaStream_t st) {
    OmParams q;
    q.a = a;
    q.b = b;
    q.len = len;
    q.na = na;
    q.nb = nb;
    q.sym = sym ? 1 : 0;
    q.brow = sym ? 0 : na;
    q.tiles_j = (nb + OM_N - 1) / OM_N;
    long long tiles = 0;
    om_shape(na, nb, len, sym, q.nsplit, q.kper, tiles);
    int* const rexp = static_cast<int*>(ws);
    q.rexp = rexp;
    const size_t rows = (size_t)na + (sym ? 0 : nb);
    q.part = reinterpret_cast<longlong2*>(static_cast<char*>(ws) + align16(rows * q.nsplit * sizeof(int)));
    return prec == WVL_F32 ? run_om<float>(q, tiles, rexp, S, st) : run_om<double>(q, tiles, rexp, S, st);
}

cudaError_t overlap_take_timeouts(unsigned* count) {
    unsigned v = 0, z = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_om_timeouts, sizeof v);
    if (e != cudaSuccess) return e;
    if (v) e = cudaMemcpyToSymbol(g_om_timeouts, &z, sizeof z);
    *count += v;
    return e;
}

}  // namespace wvl
