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
// dropped diagonals s >= 7 (below 2^-53 of one product of the largest magnitudes per
// coefficient) and one FP64 addition per slice -- no rounding per term, which an
// FP64 sum of len terms has.
//
// These errors are relative to the rows' largest magnitudes, not to the terms of an
// entry.  Where the large values of two rows do not meet (peaks apart, tails), the
// terms could be below them, so the sum of the magnitudes |a_k b_k| is formed
// beside the digits (one more plane, FP16 values of 11 bits down to 2^-23 of the largest), and the
// reduction keeps an entry only if its error is certainly below min(len, 256) 2^-53 of
// that sum.  The other entries, and those of rows with an infinity or a NaN, which have no
// scale, are summed by FP64 products, as before the digits (overlap_sum_kernel).  Uniform
// and normal coefficients pass; 256 FP32 rows of Gaussians a tenth of their length wide all
// over it are nearly all summed in FP64: 61.6 ms (72.4 without digits).
//
// Bound: the FP64 FMA loop this replaces runs on a pipe of 1.7 lanes per clock and SM.
// Here a CTA (one per SM) owns 128 x 64 entries and a slice of k and walks it in
// stages of 32 k: 12 warps slice into the digit planes (K-major core matrices, two
// stages in shared memory) while the MMAs of the stage before, issued by one
// thread of another warp, run: per 16 k, digit q of a against digits 0 .. 6 - q of b
// side by side along N, 28 pairs in 10 instructions, and one of magnitudes.  All 16 warps
// read the accumulators.  256 FP32 vectors of 884736 coefficients, symmetric: 72.4 -> 2.8 ms
// (2.6 without the magnitudes; the FP64 loop's error of 4.4e-14, relative to the whole matrix,
// becomes 2.1e-15); 4 vectors: 1640 -> 364 us; 16 of 1024 coefficients 79 -> 32.  The MMAs issued by one of the slicing warps measured 4.1 ms (an issue
// blocks while the queue is full, and the warp's stage waits for it).  What is left:
// the tensor cores are busy for about 45 % of the time, the rest is the slicing of a
// stage (the warps' issue slots) and the reading of the accumulators, during which
// they idle.
#include <algorithm>
#include <atomic>
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
constexpr int OM_P = OM_D + 1;            // planes: the digits and the magnitudes
constexpr int OM_LBOA = OM_M * 16 + 64, OM_LBOB = OM_P * OM_N * 16 + 64;
constexpr int OM_APL = OM_CH * OM_LBOA;   // a plane of a
constexpr int OM_ABYTES = OM_P * OM_APL, OM_STAGE = OM_ABYTES + OM_CH * OM_LBOB;
constexpr int OM_SMEM = 2 * OM_STAGE;
constexpr int OM_SLOTS = 152;             // CTAs resident at once (one per SM)
static_assert(7LL * OM_KC * (1 << 14) < (1 << 24), "exact partial sums");
static_assert(OM_P * OM_N <= 512 && OM_SMEM <= 227 * 1024, "tensor and shared memory");
// the accuracy rule (om_exact_enough): an entry's error stays below OM_C 2^-53 sum |a_k b_k|
constexpr int OM_C = 256;
constexpr int OM_ZERO = -0x4000;          // exponent of a slice of zeros
// most bytes of partials (or those of one slice)
constexpr long long OM_PART = 32LL << 20;

// an entry's sum over a slice: hi 2^32 + lo, hi from the diagonals 0..2; the sum of magnitudes
struct __align__(16) OmPart {
    long long hi;
    unsigned lo;
    float mag;
};

struct OmParams {
    const void* a;
    const void* b;
    OmPart* part;        // [nsplit][na][nb]
    unsigned char* flag; // [na][nb]: entries for overlap_sum_kernel
    int* count;          // its blocks per tile that are done
    const int* rexp;     // [rows][nsplit] largest biased exponents: rows of a, then of b
    long long len, kper;
    int na, nb, nsplit, tiles_j, sym;
    int brow;            // first row of b in rexp (0 when a is b)
};

template <typename T> struct Bits;
template <> struct Bits<float> {
    static constexpr int EMAX = 255, BIAS = 181;      // x = X 2^(E - BIAS)
    // magnitudes as integers of the same order, 0 for zero only; the exponent of one
    __device__ static int mag(float x) { return (int)(__float_as_uint(x) & 0x7fffffffu); }
    // (FP32 subnormals have scales of their own, exponents 0 to -22)
    __device__ static int expo(int m) { return m >> 23 ? m >> 23 : 9 - __clz(m); }
};
template <> struct Bits<double> {
    static constexpr int EMAX = 2047, BIAS = 1077;
    __device__ static int mag(double x) {
        return max(__double2hiint(x) & 0x7fffffff, __double2loint(x) != 0 ? 1 : 0);
    }
    __device__ static int expo(int m) { return max(1, m >> 20); }
};

// X + 0x80808080808080 for X = round(x 2^(BIAS - E)), E the row's largest
// biased exponent (FP64 subnormals count as exponent 1 without the hidden bit)
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
// the digits
template <int NP>
__device__ __forceinline__ void digits_of(const unsigned (&p)[NP], __half2 (&w)[NP]) {
    const __half2 off = __halves2half2(__ushort_as_half((unsigned short)0x6480),
                                       __ushort_as_half((unsigned short)0x6480));
    #pragma unroll
    for (int i = 0; i < NP; ++i) w[i] = __hsub2(*reinterpret_cast<const __half2*>(&p[i]), off);
}
// stored as one 16- or 8-byte word
template <int NP>
__device__ __forceinline__ void put_plane(unsigned char* dst, const __half2 (&w)[NP]) {
    const unsigned* u = reinterpret_cast<const unsigned*>(&w[0]);
    if constexpr (NP == 4) *reinterpret_cast<uint4*>(dst) = make_uint4(u[0], u[1], u[2], u[3]);
    else *reinterpret_cast<uint2*>(dst) = make_uint2(u[0], u[1]);
}
// digit q of a plane's pairs, stored, and the value of the digits so far: d0 + d1 / 256 +
// d2 / 65536 in FP16 (11 bits of the value down to 2^-23 of the largest)
template <int NP>
__device__ __forceinline__ void put_digits(unsigned char* dst, int q, const unsigned (&p)[NP], __half2 (&m)[NP]) {
    __half2 w[NP];
    digits_of(p, w);
    put_plane(dst, w);
    if (q > 2) return;
    const __half2 sc = __float2half2_rn(q == 1 ? 0x1p-8f : 0x1p-16f);
    #pragma unroll
    for (int i = 0; i < NP; ++i) m[i] = q == 0 ? w[i] : __hfma2(w[i], sc, m[i]);
}
template <int NP>
__device__ __forceinline__ void put_magnitudes(unsigned char* dst, __half2 (&m)[NP]) {
    #pragma unroll
    for (int i = 0; i < NP; ++i) m[i] = __habs2(m[i]);
    put_plane(dst, m);
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
    __half2 v16[NV / 2];
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
        put_digits<NV / 2>(dst + q * pl, q, p, v16);
    }
    put_magnitudes<NV / 2>(dst + OM_D * pl, v16);
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
    __half2 v16[NV / 2];
    #pragma unroll
    for (int i = 0; i < NV / 2; ++i) p[i] = __byte_perm(hi[2 * i], hi[2 * i + 1], 0x7632) + 0x64006400u;
    put_digits<NV / 2>(dst, 0, p, v16);
    #pragma unroll
    for (int w = 0; w < 3; ++w) {   // digits 1, 2 from the high word, 3 .. 6 from the low one
        #pragma unroll
        for (int i = 0; i < NV / 2; ++i)
            g[i] = w == 0 ? __byte_perm(hi[2 * i], hi[2 * i + 1], 0x5410)
                          : __byte_perm(lo[2 * i], lo[2 * i + 1], w == 1 ? 0x7632 : 0x5410);
        #pragma unroll
        for (int i = 0; i < NV / 2; ++i) p[i] = __byte_perm(g[i], H, 0x4341);
        put_digits<NV / 2>(dst + (2 * w + 1) * pl, 2 * w + 1, p, v16);
        #pragma unroll
        for (int i = 0; i < NV / 2; ++i) p[i] = __byte_perm(g[i], H, 0x4240);
        put_digits<NV / 2>(dst + (2 * w + 2) * pl, 2 * w + 2, p, v16);
    }
    put_magnitudes<NV / 2>(dst + OM_D * pl, v16);
}

// largest biased exponent of a row's slice: its scale (any, for a slice of zeros)
__device__ __forceinline__ int row_exp(const OmParams& q, int row, int split) {
    const int e = q.rexp[(long long)row * q.nsplit + split];
    return e == OM_ZERO ? 1 : e;
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
                e = max(max(e, max(Bits<T>::mag(f.x), Bits<T>::mag(f.y))),
                        max(Bits<T>::mag(f.z), Bits<T>::mag(f.w)));
            } else {
                const double2 f = __ldg(reinterpret_cast<const double2*>(x + k));
                e = max(e, max(Bits<T>::mag(f.x), Bits<T>::mag(f.y)));
            }
        }
    } else {
        #pragma unroll 4
        for (long long k = k0 + threadIdx.x; k < k1; k += 256) e = max(e, Bits<T>::mag(x[k]));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) e = max(e, red[w]);
        rexp[(long long)r * q.nsplit + blockIdx.x] = e == 0 ? OM_ZERO : Bits<T>::expo(e);
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
                // the magnitudes, over the whole slice
                #pragma unroll
                for (int ks = 0; ks < OM_KS / 16; ++ks)
                    mma(tm + OM_D * OM_N, ad + (uint64_t)((OM_D * OM_APL + 2 * ks * OM_LBOA) >> 4),
                        bd + (uint64_t)((2 * ks * OM_LBOB + OM_D * OM_N * 16) >> 4), idesc_f16(OM_M, OM_N),
                        (st == 0 && ks == 0) ? 0u : 1u);
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
    if (ok) {
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            // (the last accumulation's commit covers the magnitudes' MMAs too)
            uint32_t mg[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            if (nst > 0) {
                fence_after();
                tld8(tl + OM_D * OM_N + 8 * h, mg);
                tld_wait();
            }
            if (i0 + er >= q.na) continue;
            OmPart* const P = q.part + ((long long)blockIdx.x * q.na + i0 + er) * q.nb + j0 + ec + 8 * h;
            #pragma unroll
            for (int c = 0; c < 8; ++c)
                if (j0 + ec + 8 * h + c < q.nb) {
                    OmPart v;
                    v.hi = hi[8 * h + c];
                    v.lo = lo[8 * h + c];
                    v.mag = __uint_as_float(mg[c]);
                    P[c] = v;
                }
        }
    }
    fence_before();
    __syncthreads();
    if (tid == 0 && dead) atomicAdd(&g_om_timeouts, 1u);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tm), "r"(512));
}

// S[i][j] = the slices' integers, each scaled, added in a fixed order by rl lanes
// (one lane walking 152 slices is a chain of loads that took 40 us); when symmetric, the
// entries below the diagonal are those above it.  flag: entries of a row without a scale
// (infinity or NaN), and those whose digits may not be accurate enough.  A slice's error
// is below 8 2^-42 per coefficient in units of the digits' scale (|y| < 128: the six
// dropped products of diagonal 7, 6 2^14 2^-56, and the roundings of both inputs, 2^-49 of
// the other's magnitude), so
//   error <= sum_slices 2^-39 len_s scale_s <= OM_C 2^-53 sum_s mag_s scale_s
// holds where the magnitudes' sums say so; a row that is zero in a slice has no error there.
// For rows of fewer coefficients than OM_C the factor is their number, as an FP64 sum has.
template <typename T>
__global__ void __launch_bounds__(256) overlap_mma_reduce_kernel(const OmParams q, int rl, int tiles,
                                                                 double* __restrict__ S) {
    const long long n = (long long)q.na * q.nb;
    const int EB = 256 / rl;   // entries per block and turn
    for (int t = blockIdx.x * 256 + threadIdx.x; t < tiles; t += gridDim.x * 256) q.count[t] = 0;
    const float need = 16384.f * 1.0625f / (float)min(q.len, (long long)OM_C);
    #pragma unroll 1
    for (long long base = (long long)blockIdx.x * EB; base < n; base += (long long)gridDim.x * EB) {
        const int part = threadIdx.x % rl;
        const long long e = base + threadIdx.x / rl;
        int top = 2 * OM_ZERO, bad = 0, i = 0, j = 0;   // top: the largest scale
        if (e < n) {
            i = (int)(e / q.nb);
            j = (int)(e - (long long)i * q.nb);
            if (q.sym && i > j) { const int u = i; i = j; j = u; }
            #pragma unroll 4
            for (int s = part; s < q.nsplit; s += rl) {
                const int Ea = q.rexp[(long long)i * q.nsplit + s];
                const int Eb = q.rexp[(long long)(q.brow + j) * q.nsplit + s];
                bad |= Ea == Bits<T>::EMAX || Eb == Bits<T>::EMAX;
                if (Ea != OM_ZERO && Eb != OM_ZERO) top = max(top, Ea + Eb);
            }
        }
        #pragma unroll 1
        for (int off = rl / 2; off > 0; off >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, off, rl));
        double t = 0.0;
        float mag = 0.f, err = 0.f;
        if (e < n) {
            #pragma unroll 4
            for (int s = part; s < q.nsplit; s += rl) {
                const int Ea = q.rexp[(long long)i * q.nsplit + s];
                const int Eb = q.rexp[(long long)(q.brow + j) * q.nsplit + s];
                if (Ea == OM_ZERO || Eb == OM_ZERO) continue;
                const OmPart v = q.part[(long long)s * n + (long long)i * q.nb + j];
                // x 2^32 + y, in units of 2^48 of the integers' product
                t += scalbn(fma((double)v.hi, 4294967296.0, (double)v.lo), 48 + Ea + Eb - 2 * Bits<T>::BIAS);
                const float sc = ldexpf(1.f, Ea + Eb - top);
                mag = fmaf(v.mag, sc, mag);
                err = fmaf((float)(min(q.len, (s + 1) * q.kper) - s * q.kper), sc, err);
            }
        }
        #pragma unroll 1
        for (int off = rl / 2; off > 0; off >>= 1) {
            t += __shfl_down_sync(0xffffffffu, t, off, rl);
            mag += __shfl_down_sync(0xffffffffu, mag, off, rl);
            err += __shfl_down_sync(0xffffffffu, err, off, rl);
            bad |= __shfl_down_sync(0xffffffffu, bad, off, rl);
        }
        if (e < n && part == 0) {
            S[e] = t;
            q.flag[e] = bad || !(mag >= need * err);
        }
    }
}

// The entries that the digits do not serve, by FP64 products and sums: tiles of 32 x 32
// entries, slices of k staged in shared memory as doubles, 2 x 2 entries per thread, partials
// per slice; a tile's last block adds them in order.  Tiles without a flag end at once
// (all: every entry; small calls come here directly).  The products fill the
// FP64 pipe (1.7 lanes per clock and SM): 72.4 ms for all entries of 256 FP32 vectors of 884736
// coefficients, against 2.6 ms by digits.
constexpr int OS_T = 32, OS_KC = 64, OS_RS = OS_KC + 1;
template <typename T>
__global__ void __launch_bounds__(256) overlap_sum_kernel(const OmParams q, double* __restrict__ part, int nsplit,
                                                          long long kper, int all, double* __restrict__ S) {
    __shared__ double As[OS_T * OS_RS], Bs[OS_T * OS_RS];
    const int tj_n = (q.nb + OS_T - 1) / OS_T;
    int ti, tj;
    if (q.sym) {   // row by row, tj >= ti
        int r = blockIdx.y, t = 0;
        while (r >= tj_n - t) { r -= tj_n - t; ++t; }
        ti = t;
        tj = t + r;
    } else {
        ti = blockIdx.y / tj_n;
        tj = blockIdx.y - ti * tj_n;
    }
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, i0 = ti * OS_T, j0 = tj * OS_T;
    bool mine[2][2];
    #pragma unroll
    for (int r = 0; r < 2; ++r)
        #pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int i = i0 + 2 * ty + r, j = j0 + 2 * tx + c;
            mine[r][c] = i < q.na && j < q.nb && (all || q.flag[(long long)i * q.nb + j]);
        }
    if (!__syncthreads_or(mine[0][0] || mine[0][1] || mine[1][0] || mine[1][1])) return;
    const T* const A = static_cast<const T*>(q.a);
    const T* const B = static_cast<const T*>(q.b);
    const long long k0 = blockIdx.x * kper, k1 = min(q.len, k0 + kper);
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    #pragma unroll 1
    for (long long kb = k0; kb < k1; kb += OS_KC) {
        for (int e = threadIdx.x; e < OS_T * OS_KC; e += 256) {
            const int row = e / OS_KC, kk = e - row * OS_KC;
            const long long k = kb + kk;
            As[row * OS_RS + kk] = i0 + row < q.na && k < k1 ? (double)A[(i0 + row) * q.len + k] : 0.0;
            Bs[row * OS_RS + kk] = j0 + row < q.nb && k < k1 ? (double)B[(j0 + row) * q.len + k] : 0.0;
        }
        __syncthreads();
        #pragma unroll 8
        for (int kk = 0; kk < OS_KC; ++kk) {
            const double a0 = As[(2 * ty) * OS_RS + kk], a1 = As[(2 * ty + 1) * OS_RS + kk];
            const double b0 = Bs[(2 * tx) * OS_RS + kk], b1 = Bs[(2 * tx + 1) * OS_RS + kk];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
        __syncthreads();
    }
    const long long n = (long long)q.na * q.nb;
    if (nsplit > 1) {
        #pragma unroll
        for (int r = 0; r < 2; ++r)
            #pragma unroll
            for (int c = 0; c < 2; ++c)
                if (mine[r][c]) part[blockIdx.x * n + (long long)(i0 + 2 * ty + r) * q.nb + j0 + 2 * tx + c] = acc[r][c];
        __shared__ int last;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(q.count + blockIdx.y, 1) == nsplit - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
    }
    #pragma unroll
    for (int r = 0; r < 2; ++r)
        #pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (!mine[r][c]) continue;
            const long long i = i0 + 2 * ty + r, j = j0 + 2 * tx + c;
            double s = acc[r][c];
            if (nsplit > 1) {
                s = 0.0;
                #pragma unroll 4
                for (int p = 0; p < nsplit; ++p) s += __ldcg(part + p * n + i * q.nb + j);
            }
            // (a diagonal tile holds both halves; its lower one takes the upper's value)
            if (!q.sym || i <= j) S[i * q.nb + j] = s;
            if (q.sym && i < j) S[j * q.nb + i] = s;
        }
}

// Slices of k: whole accumulations of OM_KC, as many as minimise the waves of
// CTAs (one per SM) times a slice's length, each CTA costing about four
// accumulations more (start, exponents, partials), as long as their partials stay within
// OM_PART (16 bytes per entry and slice: waves alone asked for 304 MB at 1000 vectors for
// 4 %).  The same on every GPU, so that the workspace bound holds.
// a slice's high integer takes 2^41 per accumulation
long long om_min_slices(long long chunks) { return (chunks + (1 << 21) - 1) >> 21; }
long long om_max_slices(int na, int nb, long long len) {
    const long long chunks = std::max(1LL, (len + OM_KC - 1) / OM_KC);
    const long long most = std::max(1LL, OM_PART / ((long long)sizeof(OmPart) * na * nb));
    return std::max(om_min_slices(chunks), std::min({chunks, 2LL * OM_SLOTS, most}));
}
void om_shape(int na, int nb, long long len, bool sym, int& nsplit, long long& kper, long long& tiles) {
    const long long ti = (na + OM_M - 1) / OM_M, tj = (nb + OM_N - 1) / OM_N;
    tiles = sym ? ti * tj - ti * (ti - 1) : ti * tj;
    const long long chunks = std::max(1LL, (len + OM_KC - 1) / OM_KC);
    long long best = -1, ns = 1;
    for (long long s = om_min_slices(chunks), e = om_max_slices(na, nb, len); s <= e; ++s) {
        const long long cost = (tiles * s + OM_SLOTS - 1) / OM_SLOTS * ((chunks + s - 1) / s + 4);
        if (best < 0 || cost < best) {
            best = cost;
            ns = s;
        }
    }
    kper = (chunks + ns - 1) / ns * OM_KC;
    nsplit = (int)((chunks * OM_KC + kper - 1) / kper);
}

// Tiles and slices of overlap_sum_kernel: about four blocks per SM, slices of at least four
// stages, their partials where those of the digits were.
int os_tiles(int na, int nb, bool sym) {
    const int ti = (na + OS_T - 1) / OS_T, tj = (nb + OS_T - 1) / OS_T;
    return sym ? ti * (ti + 1) / 2 : ti * tj;
}
void os_shape(long long len, int tiles, int most, int& nsplit, long long& kper) {
    long long ns = std::max(1LL, (4LL * OM_SLOTS + tiles - 1) / tiles);
    ns = std::min({ns, std::max(1LL, len / (4 * OS_KC)), (long long)most});
    kper = std::max(1LL, ((len + ns - 1) / ns + OS_KC - 1) / OS_KC) * OS_KC;
    nsplit = (int)std::max(1LL, (len + kper - 1) / kper);
}

template <typename T>
cudaError_t om_prepare() {
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load() & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(overlap_mma_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, OM_SMEM);
    if (e == cudaSuccess) done.fetch_or(bit);
    return e;
}

template <typename T>
cudaError_t run_os(const OmParams& q, int stiles, int most, bool all, double* S, cudaStream_t st) {
    int ns = 1;
    long long kper = 0;
    os_shape(q.len, stiles, most, ns, kper);
    overlap_sum_kernel<T><<<dim3((unsigned)ns, (unsigned)stiles), 256, 0, st>>>(
        q, reinterpret_cast<double*>(q.part), ns, kper, all ? 1 : 0, S);
    count_launches(1);
    return cudaGetLastError();
}

template <typename T>
cudaError_t run_om(const OmParams& q, long long tiles, int* rexp, double* S, cudaStream_t st) {
    const int stiles = os_tiles(q.na, q.nb, q.sym);
    // one stage of FP64 sums in one wave of blocks: a single launch (64 vectors of 64
    // coefficients 24 us with the host's part, 28 by digits; of 256 coefficients 82 and 30)
    if (q.len <= OS_KC && stiles <= 4 * OM_SLOTS) return run_os<T>(q, stiles, 1, true, S, st);
    cudaError_t e = om_prepare<T>();
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
    overlap_mma_reduce_kernel<T><<<(unsigned)blocks, 256, 0, st>>>(q, rl, stiles, S);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return run_os<T>(q, stiles, 2 * q.nsplit, false, S, st);
}

size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// exponents, partials, flags, counters
size_t om_bytes(int na, int nb, size_t rows, long long ns, size_t parts) {
    const size_t tiles = (size_t)((na + OS_T - 1) / OS_T) * ((nb + OS_T - 1) / OS_T);
    return align16(rows * ns * sizeof(int)) + parts + align16((size_t)na * nb) + tiles * sizeof(int);
}

}  // namespace

size_t overlap_mma_ws(int na, int nb, long long len, bool sym) {
    int ns = 1;
    long long kper = 0, tiles = 0;
    om_shape(na, nb, len, sym, ns, kper, tiles);
    return om_bytes(na, nb, (size_t)na + (sym ? 0 : nb), ns, (size_t)ns * na * nb * sizeof(OmPart));
}
// Enough for every call of at most these sizes: grows with each of them (the slices of a call
// do not: more rows, fewer slices)
size_t overlap_mma_ws_bound(int na, int nb, long long len) {
    const long long chunks = std::max(1LL, (len + OM_KC - 1) / OM_KC);
    const long long ns = std::max(om_min_slices(chunks), std::min(chunks, 2LL * OM_SLOTS));
    const size_t one = (size_t)na * nb * sizeof(OmPart);
    const size_t parts = std::max(one * (size_t)om_min_slices(chunks),
                                  std::min(one * (size_t)ns, std::max((size_t)OM_PART, one)));
    return om_bytes(na, nb, (size_t)na + nb, ns, parts);
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
    char* w = static_cast<char*>(ws);
    int* const rexp = reinterpret_cast<int*>(w);
    q.rexp = rexp;
    w += align16(((size_t)na + (sym ? 0 : nb)) * q.nsplit * sizeof(int));
    q.part = reinterpret_cast<OmPart*>(w);
    w += (size_t)q.nsplit * na * nb * sizeof(OmPart);
    q.flag = reinterpret_cast<unsigned char*>(w);
    q.count = reinterpret_cast<int*>(w + align16((size_t)na * nb));
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
