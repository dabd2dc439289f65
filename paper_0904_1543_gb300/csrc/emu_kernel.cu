// The emulated FP64 pass (see emu.cuh for the arithmetic) as a tcgen05
// kernel for sm_103a.
//
// A window is 128 lines x 16 outputs reading 32 input positions, two 16-position
// slabs (the kinetic filter 48, three).  A work unit is a whole 128-line tile of
// one orbital (of each orbital of a group in turn in the potential pass, whose
// density partial it updates in place), walked window by window.  A persistent CTA of
// 256 threads, three per SM (two in the kinetic passes), per window
//   1. slices the window's new slab: reads it from the copies that its threads made
//      under the window before (cp.async, wrapped periodically; synthesis pass 1
//      gathers from the compressed layout instead), puts every line on its
//      scale, and writes six FP16 digit planes into a ring of slab slots
//      in shared memory, in the MMA's K-major layout (8 x 16 B core matrices);
//   2. issues, from one thread, 6 data digits x 2 or 3 K-steps of MMAs
//      (M = 128, K = 16), each over the filter digits side by side along N,
//      adding the 26 digit pairs' products into seven FP32 accumulators
//      (one per diagonal, N columns each) in tensor memory, and commits them
//      to an mbarrier, polled with a bound; meanwhile every thread loads the
//      epilogue's other inputs;
//   3. reads the accumulators (warp w: lines 32 (w % 4) + lane, half of the
//      outputs), recombines them into 64-bit integers and runs the pass's
//      epilogue (transposed store, compressed scatter, V psi with density
//      and Epot, kinetic K_p and Ekin).
// Between the passes of one operator the outputs stay these integers, with a scale per
// line (Seg::gout): the next pass shifts them to its own line's scale, the exponent of the
// line's largest element, without a scan of its inputs, and the FP64 pipe
// (a conversion and a multiplication per output otherwise) is left out.  The producing warps
// note that exponent per line of the next pass as they store (warp_tops, emu.cuh: hand_slots).
// Where an FP64 array comes in, a line's exponent is the largest of a first read.
// One scale for all lines that cross the same source lines would do without the notes and
// the shifts to the left (23.6 ms instead of 24.9 per headline step), but lines
// far below their neighbours then lose their bits (a Gaussian of 2.5 points, modelled: at 1e-6
// of its peak off two axes, 2e-12 of the element instead of 6e-15).  H psi of random coefficients:
// 1.2e-16 in the 2-norm (FP64 kernels 4.2e-16).
// Per headline step (192 orbitals): 30.9 ms with windows of 32 outputs, two CTAs per SM;
// 29.2 with 16 outputs and three; 28.5 with fields masked and completed in one
// operation; 24.7 with the integers and the copies, 23.6 with the kinetic passes' rows,
// 24.9 with a scale per line (integers and copies: neither alone gains,
// without the scan's first read the slabs' loads wait for HBM, and copies of FP64 arrays leave
// the scan; an L2 prefetch of the next slab gave 27.5, of the next tile 29.4, a
// register prefetch of the next slab 31.7).
// The filter digit planes are built once per CTA from the launch's taps.
#include <cmath>
#include <type_traits>

#include <cuda_fp16.h>

#include "emu.cuh"
#include "pass_kernel.cuh"
#include "tcgen05.cuh"

namespace wvl {

__device__ unsigned int g_emu_timeouts = 0;

namespace emu {

using namespace tc;

enum { IO_IN = 1, IO_OUT = 2 };   // integer input, output of a pass

// a b + c, 32 x 32 + 64 bits
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// input value at position x (0 <= x < n) of line a of orbital orb
template <int MODE>
__device__ __forceinline__ double load_in(const Seg<double>& S, int orb, int a, int x) {
    if (MODE == M_UNCOMP) {
        // line a = (x3, x2) of the interleaved coarse array: element x is
        // c^mu[x3/2][x2/2][x/2], mu = (x & 1) + 2 (x2 & 1) + 4 (x3 & 1)
        const int x3 = a / S.N2, x2 = a - x3 * S.N2;
        const int mu = (x & 1) + 2 * (x2 & 1) + 4 * (x3 & 1);
        const double* cc = S.in + (long long)orb * S.clen;
        const long long ci = ((long long)(x3 >> 1) * S.n2 + (x2 >> 1)) * S.n1 + (x >> 1);
        if (S.mapc == nullptr && S.bx1 == 0)
            return (mu == 0) ? cc[ci] : cc[S.ncoarse + ci * 7 + mu - 1];
        const int k = stored_index(S, ci, x >> 1, x2 >> 1, x3 >> 1, mu);
        if (k < 0) return 0.0;
        return (mu == 0) ? cc[k] : cc[S.ncoarse + (long long)k * 7 + mu - 1];
    }
    return S.in[(long long)orb * S.P + (long long)a * S.n + x];
}

// One job: orbital orb of work unit u (line tile x output window).
struct EJob {
    long long u;
    int si, grp, tt, a0, o, lt, orb, oe;
    bool valid;
};

__device__ __forceinline__ void decode_unit(const PassParams<double>& p, int mode, EJob& J) {
    J.valid = J.u < p.nunits;
    if (!J.valid) return;
    int si = 0;
    while (si + 1 < p.nseg && J.u >= p.seg[si + 1].blk0) ++si;
    const Seg<double>& S = p.seg[si];
    const long long loc = J.u - S.blk0;
    J.si = si;
    J.grp = (int)(loc / S.tiles);
    J.tt = (int)(loc - (long long)J.grp * S.tiles);
    // unit = (orbital, or orbital group in the potential pass) x a whole
    // tile of lines; the kernel walks the tile's windows
    J.a0 = J.tt * M;
    J.o = 0;
    J.lt = min(M, S.N - J.a0);
    if (mode == M_POT) {
        J.orb = J.grp * S.opg;
        J.oe = min(S.norb, J.orb + S.opg);
    } else {
        J.orb = J.grp;
        J.oe = J.grp + 1;
    }
}
__device__ __forceinline__ void first_job(const PassParams<double>& p, int mode, EJob& J) {
    J.u = blockIdx.x;
    decode_unit(p, mode, J);
}
// returns true when J was the last orbital of its unit
__device__ __forceinline__ bool next_job(const PassParams<double>& p, int mode, EJob& J) {
    if (J.orb + 1 < J.oe) {
        ++J.orb;
        return false;
    }
    J.u += gridDim.x;
    decode_unit(p, mode, J);
    return true;
}

// The 26 digit pairs of the canonical schedule (diagonal d = 2..8, i.e.
// dq + fp = d - 2 <= 6, accumulating in tensor-memory columns (d - 2) N..)
// as 6 data digits x 2 K-steps (3 for the kinetic filter): the MMA of data digit dq multiplies it by the
// filter digits fp = 0 .. 6 - dq side by side (N (7 - dq) columns from column
// dq N), so one instruction adds the products of every pair with that dq to
// their diagonals.  The first one (dq = 0, K-step 0) also meets the zero
// block (fp = 6) and so starts all seven accumulators.  Every exact
// diagonal's partial sums stay integers below 2^24 in any order, so the
// order of the pairs does not change the result.  K-step k reads the data
// planes' slab slot (slot0 + k) mod the number of K-steps; the shared-memory descriptors are base
// + compile-time offsets.
template <int KIND, int MODE>
__device__ __forceinline__ void issue_window_mmas(uint32_t tm, uint32_t a_base, uint32_t b_base,
                                                  int slot0) {
    constexpr int LBOA = lboa(MODE);
    constexpr int APL = plane_a_bytes(KIND, MODE);
    constexpr int N = window_n(KIND), LBOB = lbo_b(KIND), K = window_k(KIND);
    static_assert(S == 6 && DMAX - 2 == S, "one block per filter digit plus the zero block");
    const uint64_t a0d = mdesc(a_base, LBOA, 128), b0d = mdesc(b_base, LBOB, 128);
    uint32_t aoff[K / 16];
#pragma unroll
    for (int k = 0; k < K / 16; ++k) {
        int sl = slot0 + k;
        sl -= (sl >= K / 16) ? K / 16 : 0;
        aoff[k] = (uint32_t)(sl * 2 * LBOA) >> 4;
    }
#pragma unroll
    for (int dq = 0; dq < S; ++dq) {
        const uint32_t idesc = idesc_f16(M, N * (S + 1 - dq));
#pragma unroll
        for (int k = 0; k < K / 16; ++k)
            mma(tm + dq * N, a0d + (uint64_t)(((uint32_t)(dq * APL) >> 4) + aoff[k]),
                b0d + (uint64_t)((2 * k * LBOB) >> 4), idesc, (dq == 0 && k == 0) ? 0u : 1u);
    }
}

// The epilogue's other inputs for this thread's outputs (line er, outputs
// o0 .. o0 + N/2 - 1), loaded while the MMAs run: the kinetic passes' K_{p-1}
// (line-major, 16-byte loads) and K_0; the potential pass's V.
template <int KIND, int MODE>
__device__ __forceinline__ void prefetch_epilogue(const Seg<double>& Sg, int o0, int er, int lt,
                                                  int a0, int orb, int grp,
                                                  double (&pa)[window_n(KIND) / 2],
                                                  double (&pb)[window_n(KIND) / 2],
                                                  double (&pc)[window_n(KIND) / 2]) {
    constexpr int NH = window_n(KIND) / 2;
    constexpr bool KM = (MODE == M_KMID || MODE == M_KLAST);
    if (!(KM || MODE == M_POT)) return;
    const int n = Sg.n, NL = Sg.N;
    const int a = a0 + er;
    const long long obase = (long long)orb * Sg.P;
    const bool full = er < lt && o0 + NH <= n;   // all outputs exist: vector loads
#pragma unroll
    for (int c = 0; c < NH; ++c) {
        if (!KM) pa[c] = 0.0;   // (the kinetic passes' G is there already)
        pb[c] = pc[c] = 0.0;
    }
    if (er >= lt) return;
    if (KM) {
        const double* ki = Sg.in2 ? Sg.in2 + obase + (long long)a * n + o0 : nullptr;
        if (ki != nullptr) {
            if (full) {
#pragma unroll
                for (int c = 0; c < NH; c += 2) {
                    const double2 k2 = *reinterpret_cast<const double2*>(ki + c);
                    pb[c] = k2.x;
                    pb[c + 1] = k2.y;
                }
            } else {
#pragma unroll
                for (int c = 0; c < NH; ++c)
                    if (o0 + c < n) pb[c] = ki[c];
            }
        }
        if (MODE == M_KLAST && Sg.aux)
#pragma unroll
            for (int c = 0; c < NH; ++c)
                if (o0 + c < n) pc[c] = Sg.aux[obase + (long long)(o0 + c) * NL + a];
    } else if (MODE == M_POT) {
        if (Sg.aux)
#pragma unroll
            for (int c = 0; c < NH; ++c)
                if (o0 + c < n) pa[c] = Sg.aux[(long long)(o0 + c) * NL + a];
        // the density so far is read in the epilogue: prefetched too, it
        // would stay live across the MMAs beside V and spill
    }
}

// Where a warp writes the largest exponents of its integer outputs, per output I and line of
// the next pass (emu.cuh, hand_slots): source line a belongs to the next pass's line
// I step + a / nnext, the warp's lines to more + 1 of them per output.
struct HandOut {
    int* top;    // output 0's entry of the first line, in the warp's slot of it
    int* top0;   // the same entry in slot 0, which the others take
    int step, more;
};
// exponents as pairs of 16 bits, one pair per two outputs
__device__ __forceinline__ unsigned pair16(int a, int b) { return __byte_perm((unsigned)a, (unsigned)b, 0x5410); }
constexpr int HAND_NONE = -30000;
// The largest over the warp's lanes of every one of the eight exponents in p, handed to
// put(output, largest) by one lane each: half of the pairs go across in each of the first two
// exchanges, so that six shuffles do (25.0 ms per headline step; 25.9 with eight warp
// reductions and stores).
template <typename F>
__device__ __forceinline__ void warp_tops(const unsigned (&p)[4], F&& put) {
    const int lane = threadIdx.x & 31;
    const bool h = lane & 16, l = lane & 8;
    unsigned q0 = h ? p[2] : p[0], q1 = h ? p[3] : p[1];
    q0 = __vmaxs2(q0, __shfl_xor_sync(0xffffffffu, h ? p[0] : p[2], 16));
    q1 = __vmaxs2(q1, __shfl_xor_sync(0xffffffffu, h ? p[1] : p[3], 16));
    unsigned r = l ? q1 : q0;
    r = __vmaxs2(r, __shfl_xor_sync(0xffffffffu, l ? q0 : q1, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) r = __vmaxs2(r, __shfl_xor_sync(0xffffffffu, r, o));
    if ((lane & 7) < 2) put(2 * (lane >> 3) + (lane & 1), (lane & 1) ? (int)r >> 16 : (int)(short)r);
}

// one window's outputs of this thread (line er, outputs o0 .. o0 + N/2 - 1):
// accumulators -> FP64 -> the pass's epilogue; returns the energy partial
template <int KIND, int MODE, bool OUTI>
__device__ __forceinline__ double window_epilogue(const Seg<double>& Sg, uint32_t tl, int o0,
                                                  int er, int lt, int a0, int orb, int grp, int se,
                                                  const double (&pa)[window_n(KIND) / 2],
                                                  const double (&pb)[window_n(KIND) / 2],
                                                  const double (&pc)[window_n(KIND) / 2],
                                                  const HandOut* hos, const unsigned char* rowS) {
    constexpr int N = window_n(KIND), NH = N / 2;
    constexpr bool KM = (MODE == M_KMID || MODE == M_KLAST);
    const int n = Sg.n, NL = Sg.N;
    const int gl = se;   // (integer output: the line's scale)
    se = max(-1022, min(1023, se));
    // 2^se as a double: the FP64 pipe is idle here, the integer pipes are not
    const double scale = __longlong_as_double((long long)(se + 1023) << 52);
    const bool row_ok = er < lt;
    const int a = a0 + er;
    const long long obase = (long long)orb * Sg.P;
    double occ = 1.0;
    if (MODE == M_POT) occ = Sg.occ ? Sg.occ[orb] : 1.0;
    // M_COMP for the adjoint of E_loc: H psi scaled by 2 occ g
    double osc = 1.0;
    if (MODE == M_COMP && Sg.gscale != nullptr) osc = 2.0 * Sg.occ[orb] * Sg.gscale[0];
    double eacc = 0.0;
    static_assert(NH == 8 && NACC == 7 && NEXACT == 4 && DBITS == 10 && TSHIFT == 20 && DMAX == 8, "recombination");
    uint32_t dv[NACC][8];
#pragma unroll
    for (int ac = 0; ac < NACC; ++ac) tld8(tl + ac * N, dv[ac]);
    tld_wait();
    const bool full = o0 + NH <= n;   // every output exists
    // element (I, a) of the transposed output is at obase + I NL + a
    const long long oi0 = obase + (long long)o0 * NL + a;
    // M_COMP on the full grid: the outputs' positions in the compressed form, two outputs per
    // coarse point along the line (components mu12 and mu12 + 4)
    double* ce = nullptr;
    double* co = nullptr;
    long long se_ = 0, so_ = 0;
    int X1 = 0, X2 = 0;
    const bool plain = Sg.mapc == nullptr && Sg.bx1 == 0;
    if (MODE == M_COMP) {
        X2 = a / Sg.N1;
        X1 = a - X2 * Sg.N1;
        const int mu12 = (X1 & 1) + 2 * (X2 & 1);
        const int plane = Sg.n1 * Sg.n2, cx = (X2 >> 1) * Sg.n1 + (X1 >> 1);
        double* const cc0 = Sg.out + (long long)orb * Sg.clen;
        so_ = 7LL * plane;
        se_ = mu12 == 0 ? plane : so_;
        const long long i2 = o0 >> 1;
        ce = (mu12 == 0 ? cc0 + cx : cc0 + Sg.ncoarse + 7LL * cx + mu12 - 1) + i2 * se_;
        co = cc0 + Sg.ncoarse + 7LL * cx + mu12 + 3 + i2 * so_;
    }
    if (OUTI ? lt <= (er & ~31) : !row_ok) return 0.0;   // (integer output: whole warps)
    unsigned pe[NH / 2];   // exponents of the integer outputs
    {
#pragma unroll
        for (int c = 0; c < NH; ++c) {
            // diagonals 0 .. 3 (exact integers, weights 2^40 .. 2^10) and the sum of the
            // low ones (weights 1, 2^-10, 2^-20), in one 64-bit integer
            int i[NEXACT];
#pragma unroll
            for (int ac = 0; ac < NEXACT; ++ac) i[ac] = __float2int_rn(__uint_as_float(dv[ac][c]));
            float low = __uint_as_float(dv[4][c]);
            low = fmaf(__uint_as_float(dv[5][c]), 0x1p-10f, low);
            low = fmaf(__uint_as_float(dv[6][c]), 0x1p-20f, low);
            const int i01 = i[0] * 1024 + i[1];
            long long t = __float2int_rn(low);
            t = mad_wide(i[3], 1 << 10, t);
            t = mad_wide(i[2], 1 << 20, t);
            t = mad_wide(i01, 1 << 30, t);
            const int I = o0 + c;
            if (!full && I >= n) {
                if (OUTI) pe[c / 2] = c & 1 ? pair16((int)pe[c / 2], HAND_NONE) : (unsigned)HAND_NONE;
                continue;
            }
            const long long oi = oi0 + (long long)c * NL;
            if constexpr (OUTI) {
                // the next pass reads the integer, the line's scale and the largest exponent
                // of its own lines, |t| 2^gl <= 2^e (0: 2^-126 of the scale)
                const int e = gl + hand_bits(__ll2float_rn(t));
                pe[c / 2] = c & 1 ? pair16((int)pe[c / 2], e) : (unsigned)e;
                if (row_ok) reinterpret_cast<long long*>(Sg.out)[oi] = t;
                continue;
            }
            const double val = (double)t * scale;
            if (MODE == M_PLAIN || MODE == M_UNCOMP) {
                Sg.out[oi] = val;
            } else if (MODE == M_COMP) {
                const double sv = Sg.gscale != nullptr ? val * osc : val;
                if (plain) {
                    if (c & 1) co[(c >> 1) * so_] = sv;
                    else ce[(c >> 1) * se_] = sv;
                } else {
                    const int mu = (X1 & 1) + 2 * (X2 & 1) + 4 * (I & 1);
                    const long long ci = ((long long)(I >> 1) * Sg.n2 + (X2 >> 1)) * Sg.n1 + (X1 >> 1);
                    double* const cc0 = Sg.out + (long long)orb * Sg.clen;
                    const int k = stored_index(Sg, ci, X1 >> 1, X2 >> 1, I >> 1, mu);
                    if (k >= 0) {
                        if (mu == 0) cc0[k] = sv;
                        else cc0[Sg.ncoarse + (long long)k * 7 + mu - 1] = sv;
                    }
                }
            } else if (KM) {
                const double g = pa[c];
                double kin = pb[c];
                if (MODE == M_KMID && Sg.in2 == nullptr && Sg.eps != nullptr) kin = -Sg.eps[orb] * g;
                const double acc = val + kin;
                if (MODE == M_KMID) {
                    Sg.out[oi] = acc;
                    Sg.out2[oi] = g;
                } else {
                    if (Sg.out) Sg.out[oi] = acc;
                    eacc = fma(g, acc - pc[c], eacc);
                }
            } else if (MODE == M_POT) {
                if (Sg.aux) {
                    const double y = pa[c] * val;
                    if (Sg.out) Sg.out[oi] = y;
                    eacc = fma(y, val, eacc);
                }
                // the unit owns these density elements: one thread updates
                // each, orbital after orbital, in a fixed order; the density
                // so far is the caller's rho, or this group's partial after
                // the group's first orbital
                if (Sg.rho != nullptr) {
                    double* const rp = Sg.rho + (long long)grp * Sg.rho_gstride + (oi - obase);
                    const double prev = (Sg.rho_gstride == 0 || orb != grp * Sg.opg) ? *rp : 0.0;
                    *rp = fma(occ * val, val, prev);
                }
            }
        }
    }
    if constexpr (OUTI) {
        if (!row_ok)
#pragma unroll
            for (int k = 0; k < NH / 2; ++k) pe[k] = pair16(HAND_NONE, HAND_NONE);
        const HandOut ho = hos[er >> 5];
        auto tops = [&](const unsigned (&m)[NH / 2], int* top) {
            warp_tops(m, [&](int c, int e) {
                if (o0 + c < n) top[(long long)(o0 + c) * ho.step] = e;
            });
        };
        if (ho.more == 0) {
            tops(pe, ho.top);
        } else {   // the warp's lines belong to several of the next pass's
            const int seg = rowS[er];
#pragma unroll 1
            for (int k = 0; k <= ho.more; ++k) {
                unsigned m[NH / 2];
#pragma unroll
                for (int i = 0; i < NH / 2; ++i) m[i] = seg == k ? pe[i] : pair16(HAND_NONE, HAND_NONE);
                tops(m, k == 0 ? ho.top : ho.top0 + k);
            }
        }
    }
    return eacc;
}

// fixed-order CTA sum of one value per thread
__device__ __forceinline__ double cta_sum(double v, double* red) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
#pragma unroll
        for (int w = 0; w < WARPS; ++w) t += red[w];
    return t;
}

template <int KIND, int MODE, int IO>
__global__ void __launch_bounds__(THREADS, min_ctas(KIND))
emu_pass_kernel(const __grid_constant__ Params ep) {
    constexpr bool INI = (IO & IO_IN) != 0, OUTI = (IO & IO_OUT) != 0;   // integer input, output
    constexpr int K = window_k(KIND), HA = window_ha(KIND);
    constexpr int LBOA = lboa(MODE);
    constexpr int APL = plane_a_bytes(KIND, MODE);
    constexpr int NT = KT<KIND>::NT;
    constexpr int N = window_n(KIND), LBOB = lbo_b(KIND), TCOLS = tmem_cols(KIND);
    constexpr int NH = N / 2;                // outputs per epilogue thread
    constexpr int RPW = M / WARPS;           // lines per slicing warp
    constexpr int NSLOT = K / 16;            // 16-position slabs per window (3)
    static_assert(N == 16, "one new slab per window");
    extern __shared__ __align__(128) unsigned char sm[];
    unsigned char* const Asm = sm;                // [S][APL]: NSLOT slab slots of 2 chunks
    unsigned char* const Bsm = sm + S * APL;      // K / 8 chunks of (S + 1) N rows
    __shared__ uint32_t tslot;
    __shared__ __align__(8) uint64_t mbar;
    __shared__ int rowE[M];
    __shared__ int rowG[INI ? M : 1];             // integer input: a line's first source line
    __shared__ HandOut hos[OUTI ? M / 32 : 1];    // integer output
    __shared__ unsigned char rowS[OUTI ? M : 1];  // a line's line of the next pass, from its warp's first
    __shared__ double red[WARPS];

    const PassParams<double>& p = ep.p;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // ---------------------------------------------- filter digit planes
    int ebf = 0;
    for (int e = 0; e < 2; ++e)
        for (int t = 0; t < NT; ++t) ebf = max(ebf, bexp(p.f[e][t]));
    const int Ef = scale_of(ebf);
    for (int i = tid; i < N * K; i += THREADS) {
        const int j = i / K, k = i - j * K;
        const int e = j & 1;
        const int t = k - j - (HA - p.hl) - (e ? KT<KIND>::OFF1 : KT<KIND>::OFF0);
        const double f = (t >= 0 && t < NT) ? p.f[e][t] : 0.0;
        int d[S];
        digits(quantize(f, Ef), d);
        unsigned char* const b = Bsm + (k >> 3) * LBOB + j * 16 + (k & 7) * 2;
#pragma unroll
        for (int q = 0; q < S; ++q)
            *reinterpret_cast<__half*>(b + q * N * 16) = __int2half_rn(d[q]);
        *reinterpret_cast<__half*>(b + S * N * 16) = __float2half(0.f);   // the zero block
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(su32(&mbar)), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(su32(&tslot)), "r"(TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tm = tslot;
    // epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (lines)
    // and one half of the window's outputs
    const int quarter = warp & 3, half = warp >> 2;
    const int er = 32 * quarter + lane;
    const uint32_t tl = tm + ((uint32_t)(32 * quarter) << 16) + NH * half;
    const uint32_t a_base = su32(Asm), b_base = su32(Bsm);
    uint32_t phase = 0;
    bool failed = false;

    // MMAs of one window, then the wait: one thread polls, the others sleep
    // in the barrier instead of taking issue slots from the co-resident CTA
    auto issue_mmas = [&](int slot0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        fence_before();
        __syncthreads();
        if (tid == 0) {
            fence_after();
            issue_window_mmas<KIND, MODE>(tm, a_base, b_base, slot0);
            commit(su32(&mbar));
        }
    };
    auto wait_mmas = [&]() -> bool {
        bool ok = true;
        if (tid == 0) ok = wait_parity(su32(&mbar), phase);
        if (__syncthreads_or(!ok)) return false;
        phase ^= 1u;
        fence_after();
        return true;
    };

    EJob J;
    first_job(p, MODE, J);

    // The copies' cursor: the slab after the last one copied, in job Q.  A thread copies
    // exactly the 16-byte pairs that it will slice (rows r0 + 4 g, pair `pair`) and reads
    // them back itself, so its own wait is all the synchronisation they need, and they have a
    // whole window (or the previous job's last one) to arrive.
    const int pair = lane & 7, r0 = warp * RPW + (lane >> 3);
    constexpr bool ROWS = KIND == K_KIN;   // staged as whole rows, each read by the thread of its outputs
    unsigned char* const raw = sm + S * APL + b_bytes(KIND) + (ROWS ? r0 * RAWROW + pair * 16 : tid * 16);
    constexpr int RAWSTEP = ROWS ? 4 * RAWROW : THREADS * 16;
    EJob Q = J;
    const double* qsrc = nullptr;
    int qx = 0, qleft = 0, qn = 0;
    auto begin_copies = [&]() {
        if (!Q.valid) return;
        const Seg<double>& Sq = p.seg[Q.si];
        qn = Sq.n;
        qsrc = Sq.in + (long long)Q.orb * Sq.P + (long long)(Q.a0 + r0) * qn;
        qx = -HA % qn;
        if (qx < 0) qx += qn;
        qleft = Sq.nwin + NSLOT - 1;
    };
    auto copy_slab = [&]() {
        if (qleft == 0) {
            next_job(p, MODE, Q);
            begin_copies();
        }
        if (Q.valid) {
            int x = qx + 2 * pair;
            while (x >= qn) x -= qn;
#pragma unroll
            for (int g4 = 0; g4 < RPW / 4; ++g4)
                if (r0 + 4 * g4 < Q.lt) cp_async16(raw + g4 * RAWSTEP, qsrc + (long long)(4 * g4) * qn + x);
            qx += 16;
            while (qx >= qn) qx -= qn;
            --qleft;
        }
        cp_commit();
    };
    if constexpr (MODE != M_UNCOMP) {
        begin_copies();
        copy_slab();
    }
#pragma unroll 1
    while (J.valid) {
        const Seg<double>& Sg = p.seg[J.si];
        const int n = Sg.n;
        {
            // ---------------------------- one exponent per line: given (synthesis
            // pass 1 on the full grid), or the whole line read, 8 lines in flight per warp
            if constexpr (INI) {
                // the line's largest exponent, from the slots of the warps whose source lines
                // it crosses (n divides nsrc)
                if (tid < M) {
                    int e = HAND_FLOOR, a = 0;
                    if (tid < J.lt) {
                        a = (int)((unsigned)(J.a0 + tid) % (unsigned)(Sg.nsrc / n)) * n;
                        const int ns = (a + n - 1) / 32 - a / 32 + 1;
                        const int* g = Sg.gmax + (long long)J.orb * hand_slots(n) * Sg.N + J.a0 + tid;
                        for (int k = 0; k < ns; ++k, g += Sg.N) e = max(e, *g);
                    }
                    rowE[tid] = e;
                    rowG[tid] = a;
                }
            } else if (MODE == M_UNCOMP && Sg.lexp != nullptr) {
                for (int r = tid; r < M; r += THREADS)
                    rowE[r] = scale_of(r < J.lt ? Sg.lexp[(long long)J.orb * Sg.N + J.a0 + r] : 0);
            } else
#pragma unroll 1
            for (int i = 0; i < RPW; i += 8) {
                int eb[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
                for (int x = 2 * lane; x < n; x += 64) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int r = warp + WARPS * (i + k);
                        if (r >= J.lt) continue;
                        if (MODE == M_UNCOMP) {
                            eb[k] = max(eb[k], bexp(load_in<MODE>(Sg, J.orb, J.a0 + r, x)));
                            eb[k] = max(eb[k], bexp(load_in<MODE>(Sg, J.orb, J.a0 + r, x + 1)));
                        } else {
                            // n is even: x, x + 1 are in the line and 16-byte aligned
                            const double2 v = *reinterpret_cast<const double2*>(
                                Sg.in + (long long)J.orb * Sg.P + (long long)(J.a0 + r) * n + x);
                            eb[k] = max(eb[k], max(bexp(v.x), bexp(v.y)));
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)eb[k]);
                    if (lane == 0) rowE[warp + WARPS * (i + k)] = scale_of(e);
                }
            }
            __syncthreads();
            // ---------------------------- windows; each slab sliced once
            // slab s covers positions 16 s - HA .. + 15; window w reads slabs w .. w + NSLOT - 1
            // from slots (slab mod NSLOT)
            const int nwin = Sg.nwin;
            // raw inputs of one slab for this lane: lines r0 + 4 g, r0 = warp * RPW + lane / 8,
            // positions 2 (lane % 8), + 1 of the slab; with integers, their lines' scales
            struct Raw {
                long long v[RPW / 4][2];
                int g[INI ? RPW / 4 : 1][2];
            };
            const int* const gsrc = INI ? Sg.gin + (long long)J.orb * Sg.nsrc : nullptr;
            unsigned char* const adst = Asm + (pair >> 2) * LBOA + r0 * 16 + (pair & 3) * 4;
            int xs = -HA % n;            // first position of the next slab to load
            if (xs < 0) xs += n;
            int slot = 0;                // and its slot
            auto load_slab = [&](Raw& w) {
                int x = xs + 2 * pair;
                while (x >= n) x -= n;
                if constexpr (MODE != M_UNCOMP) cp_wait<0>();
#pragma unroll
                for (int g4 = 0; g4 < RPW / 4; ++g4) {
                    w.v[g4][0] = w.v[g4][1] = 0;
                    if constexpr (INI) w.g[g4][0] = w.g[g4][1] = 0;
                    if (r0 + 4 * g4 >= J.lt) continue;
                    if (MODE == M_UNCOMP) {
                        w.v[g4][0] = __double_as_longlong(load_in<MODE>(Sg, J.orb, J.a0 + r0 + 4 * g4, x));
                        w.v[g4][1] = __double_as_longlong(load_in<MODE>(Sg, J.orb, J.a0 + r0 + 4 * g4, x + 1));
                    } else {
                        // x is even and n is even: x + 1 is in the line, 16-byte aligned
                        const longlong2 d2 = *reinterpret_cast<const longlong2*>(raw + g4 * RAWSTEP);
                        w.v[g4][0] = d2.x;
                        w.v[g4][1] = d2.y;
                        if constexpr (INI) {
                            const int2 g2 = *reinterpret_cast<const int2*>(gsrc + rowG[r0 + 4 * g4] + x);
                            w.g[g4][0] = g2.x;
                            w.g[g4][1] = g2.y;
                        }
                    }
                }
                if constexpr (MODE != M_UNCOMP) copy_slab();
                xs += 16;
                while (xs >= n) xs -= n;
            };
            auto slice_slab = [&](const Raw& w) {
                unsigned char* const d = adst + slot * (2 * LBOA);
#pragma unroll
                for (int g4 = 0; g4 < RPW / 4; ++g4) {
                    const int E = rowE[r0 + 4 * g4];
                    long long y[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        if constexpr (INI) y[c] = requantize(w.v[g4][c], w.g[g4][c], E);
                        else y[c] = quantize(__longlong_as_double(w.v[g4][c]), E) + DBIAS;
                    }
                    uint32_t h[S];
                    digit_pairs(y[0], y[1], h);
#pragma unroll
                    for (int q = 0; q < S; ++q) *reinterpret_cast<uint32_t*>(d + g4 * 64 + q * APL) = h[q];
                }
                if (++slot == NSLOT) slot = 0;
            };
            if constexpr (OUTI)
                if (tid < J.lt) {
                    Sg.gout[(long long)J.orb * Sg.N + J.a0 + tid] = rowE[tid] + Ef - OUT_EXP;
                    const int nn = Sg.nnext, w0 = J.a0 + (tid & ~31);   // the warp's first source line
                    const int c0 = w0 / nn;
                    rowS[tid] = (unsigned char)((J.a0 + tid) / nn - c0);
                    if ((tid & 31) == 0) {
                        HandOut h;
                        h.step = Sg.N / nn;
                        h.more = min(w0 + 31, Sg.N - 1) / nn - c0;
                        const long long lines = (long long)n * h.step;   // of the next pass
                        h.top0 = Sg.gtop + (long long)J.orb * hand_slots(nn) * lines + c0;
                        h.top = h.top0 + (w0 / 32 - c0 * nn / 32) * lines;
                        hos[tid >> 5] = h;
                    }
                }
            // kinetic passes: the thread of line er, outputs 8 half .. + 7 of a window, slices the
            // same positions of the line's slabs, and keeps them for the epilogue: the
            // outputs of window w are the positions of slab w + 1 (pa; pn is slab w + 2)
            double pa[NH], pn[NH];
            auto row_slab = [&]() {
                cp_wait<0>();
                __syncthreads();
                const double2* const src = reinterpret_cast<const double2*>(
                    sm + S * APL + b_bytes(KIND) + er * RAWROW + half * 64);
                const int E = rowE[er];
                unsigned char* const d = Asm + (2 * slot + half) * LBOA + er * 16;
                uint32_t h[4][S];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const double2 v = er < J.lt ? src[c] : make_double2(0.0, 0.0);
                    pa[2 * c] = pn[2 * c];
                    pa[2 * c + 1] = pn[2 * c + 1];
                    pn[2 * c] = v.x;
                    pn[2 * c + 1] = v.y;
                    digit_pairs(quantize(v.x, E) + DBIAS, quantize(v.y, E) + DBIAS, h[c]);
                }
#pragma unroll
                for (int q = 0; q < S; ++q)
                    *reinterpret_cast<uint4*>(d + q * APL) = make_uint4(h[0][q], h[1][q], h[2][q], h[3][q]);
                if (++slot == NSLOT) slot = 0;
            };
            double eacc = 0.0;
            int first = 0;   // slot of the window's first slab
#pragma unroll 1
            for (int w = 0; w < nwin && !failed; ++w) {
                const int o = w * N;
                if constexpr (ROWS) {
                    if (w == 0) {
#pragma unroll 1
                        for (int k = 0; k < NSLOT; ++k) {
                            row_slab();
                            if (k + 1 < NSLOT) {
                                __syncthreads();   // the rows are read
                                copy_slab();
                            }
                        }
                    } else {
                        row_slab();
                        if (++first == NSLOT) first = 0;
                    }
                } else if (w == 0) {
#pragma unroll 1
                    for (int k = 0; k < NSLOT; ++k) {
                        Raw v;
                        load_slab(v);
                        slice_slab(v);
                    }
                } else {
                    Raw v;
                    load_slab(v);
                    slice_slab(v);
                    if (++first == NSLOT) first = 0;
                }
                issue_mmas(first);
                if constexpr (ROWS) copy_slab();   // (every row was read before the barrier above)
                double pb[NH], pc[NH];
                prefetch_epilogue<KIND, MODE>(Sg, o + NH * half, er, J.lt, J.a0, J.orb, J.grp, pa,
                                              pb, pc);

                if (!wait_mmas()) {
                    failed = true;
                    break;
                }
                eacc += window_epilogue<KIND, MODE, OUTI>(Sg, tl, o + NH * half, er, J.lt, J.a0, J.orb,
                                                    J.grp, rowE[er] + Ef - OUT_EXP, pa, pb, pc, hos, rowS);
                fence_before();
                __syncthreads();   // accumulators are rewritten by the next window's MMAs
            }
            if (failed) break;
            if (MODE == M_KLAST || (MODE == M_POT && Sg.aux)) {
                const double t = cta_sum(eacc, red);
                if (tid == 0) Sg.part[(long long)J.orb * Sg.tiles + J.tt] = t;
                __syncthreads();
            }
            __syncthreads();   // rowE and the slab ring are reused by the next job
            next_job(p, MODE, J);
        }
    }

    cp_wait<0>();
    if (failed) {
        // let the MMAs still in flight finish before the accumulators are freed
        if (tid == 0) {
            atomicAdd(&g_emu_timeouts, 1u);
            wait_parity(su32(&mbar), phase);
        }
        __syncthreads();
    }
    fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tm), "r"(TCOLS));
}

// ------------------------------------------------------------------ host
// The kernel's schedule for a launch's taps (emu.cuh: build_sched).
static bool build_sched(int kind, const PassParams<double>& p, Sched& s) {
    return emu::build_sched(p.f, kind_geom(kind).nt, s);
}

template <int KIND, int MODE, int IO>
static cudaError_t ensure_emu_attr() {
    static unsigned long long done = 0;
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(__atomic_load_n(&done, __ATOMIC_ACQUIRE) & bit)) {
        err = cudaFuncSetAttribute(emu_pass_kernel<KIND, MODE, IO>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(KIND, MODE));
        if (err != cudaSuccess) return err;
        err = cudaFuncSetAttribute(emu_pass_kernel<KIND, MODE, IO>,
                                   cudaFuncAttributePreferredSharedMemoryCarveout,
                                   cudaSharedmemCarveoutMaxShared);
        if (err != cudaSuccess) return err;
        __atomic_fetch_or(&done, bit, __ATOMIC_ACQ_REL);
    }
    return cudaSuccess;
}

template <int KIND, int MODE, int IO>
static cudaError_t launch_emu(const Params& ep, long long nunits, cudaStream_t st) {
    cudaError_t err = ensure_emu_attr<KIND, MODE, IO>();
    if (err != cudaSuccess) return err;
    if (nunits <= 0) return cudaSuccess;
    int dev = 0, nsm = 0, occ = 0;
    if ((err = cudaGetDevice(&dev)) != cudaSuccess) return err;
    if ((err = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return err;
    // CTAs per SM from shared memory, registers and tensor memory (512
    // columns); the occupancy calculator undercounts these kernels
    static int regs[64] = {0};
    if (!regs[dev & 63]) {
        cudaFuncAttributes fa;
        if ((err = cudaFuncGetAttributes(&fa, emu_pass_kernel<KIND, MODE, IO>)) != cudaSuccess) return err;
        regs[dev & 63] = std::max(fa.numRegs, 1);
    }
    int smem_sm = 0;
    if ((err = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) !=
        cudaSuccess)
        return err;
    const int per_cta = smem_bytes(KIND, MODE) + 1024 + 1024;   // + static + reserved
    const int by_smem = smem_sm / per_cta;
    const int by_regs = 65536 / (((regs[dev & 63] + 7) / 8 * 8) * THREADS);
    occ = std::min(std::min(by_smem, by_regs), 512 / tmem_cols(KIND));
    if (occ < 1) return cudaErrorInvalidConfiguration;
    long long grid = std::min<long long>((long long)occ * nsm, nunits);
    emu_pass_kernel<KIND, MODE, IO><<<dim3((unsigned)grid), dim3(THREADS), smem_bytes(KIND, MODE), st>>>(ep);
    count_launches(1);
    return cudaGetLastError();
}

// every pass kernel of the chains: f(kind, mode, io)
template <typename F>
static void for_each_emu(F&& f) {
#define EMU_K(kind, mode, io)                                                              \
    f(std::integral_constant<int, kind>{}, std::integral_constant<int, mode>{},            \
      std::integral_constant<int, io>{})
    EMU_K(K_SYN, M_UNCOMP, IO_OUT);
    EMU_K(K_ANA, M_COMP, IO_IN);
    EMU_K(K_MF, M_POT, IO_IN);
    EMU_K(K_SYN, M_PLAIN, IO_IN | IO_OUT);
    EMU_K(K_SYN, M_PLAIN, IO_IN);
    EMU_K(K_MF, M_PLAIN, IO_OUT);
    EMU_K(K_MF, M_PLAIN, IO_IN | IO_OUT);
    EMU_K(K_MF, M_PLAIN, IO_IN);
    EMU_K(K_MFT, M_PLAIN, IO_OUT);
    EMU_K(K_MFT, M_PLAIN, IO_IN | IO_OUT);
    EMU_K(K_MFT, M_PLAIN, IO_IN);
    EMU_K(K_ANA, M_PLAIN, IO_OUT);
    EMU_K(K_ANA, M_PLAIN, IO_IN | IO_OUT);
    EMU_K(K_KIN, M_KMID, 0);
    EMU_K(K_KIN, M_KLAST, 0);
#undef EMU_K
}

}  // namespace emu

// One warp per (orbital, i3, i2) row of coarse points reads the row's scaling
// coefficients and 7-component wavelet records as contiguous runs; the
// coefficient c^mu of point (i1, i2, i3) lies on line (x3, x2) = (2 i3 + a3,
// 2 i2 + a2) of the interleaved array, mu = a1 + 2 a2 + 4 a3, so the row
// gives the maxima of four lines.
__global__ void line_exp_kernel(const double* __restrict__ in, int* __restrict__ lexp, int n1,
                                int n2, int n3, long long P, long long nrows) {
    const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= nrows) return;
    const long long rows_orb = (long long)n3 * n2;
    const int orb = (int)(row / rows_orb);
    const int rem = (int)(row - orb * rows_orb);
    const int i3 = rem / n2, i2 = rem - i3 * n2;
    const double* cc = in + (long long)orb * P;
    const long long k0 = ((long long)i3 * n2 + i2) * n1;
    const double* cf = cc + P / 8 + 7 * k0;
    int m[4] = {0, 0, 0, 0};   // line (a3, a2) -> m[2 a3 + a2]
    for (int i1 = lane; i1 < n1; i1 += 32) m[0] = max(m[0], emu::bexp(cc[k0 + i1]));
    for (int pos = lane; pos < 7 * n1; pos += 32) {
        const int mu = pos % 7 + 1;
        const int e = emu::bexp(cf[pos]);
        const int l = 2 * (mu >> 2) + ((mu >> 1) & 1);
        m[0] = l == 0 ? max(m[0], e) : m[0];
        m[1] = l == 1 ? max(m[1], e) : m[1];
        m[2] = l == 2 ? max(m[2], e) : m[2];
        m[3] = l == 3 ? max(m[3], e) : m[3];
    }
#pragma unroll
    for (int l = 0; l < 4; ++l) m[l] = (int)__reduce_max_sync(0xffffffffu, (unsigned)m[l]);
    if (lane < 4) {
        const int a3 = lane >> 1, a2 = lane & 1;
        const int N2 = 2 * n2, N3 = 2 * n3;
        const int v = lane == 0 ? m[0] : lane == 1 ? m[1] : lane == 2 ? m[2] : m[3];
        lexp[(long long)orb * N2 * N3 + (long long)(2 * i3 + a3) * N2 + 2 * i2 + a2] = v;
    }
}

cudaError_t launch_line_exp(const double* in, int* lexp, int n1, int n2, int n3, int norb,
                            long long P, cudaStream_t st) {
    const long long nrows = (long long)norb * n3 * n2;
    if (nrows <= 0) return cudaSuccess;
    const int threads = 256;
    const long long blocks = (nrows * 32 + threads - 1) / threads;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    line_exp_kernel<<<(unsigned)blocks, threads, 0, st>>>(in, lexp, n1, n2, n3, P, nrows);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_pass_emu(int kind, int mode, const PassParams<double>& p, long long nunits,
                            cudaStream_t st) {
    emu::Params ep;
    std::memset(&ep, 0, sizeof ep);
    ep.p = p;
    if (!emu::build_sched(kind, p, ep.s)) return cudaErrorInvalidValue;
    using namespace emu;
    // (one launch's segments agree on integer input and output)
    const int io = (p.seg[0].gin != nullptr ? IO_IN : 0) | (p.seg[0].gout != nullptr ? IO_OUT : 0);
    cudaError_t e = cudaErrorInvalidValue;
    for_each_emu([&](auto k, auto m, auto i) {
        if (kind == k() && mode == m() && io == i()) e = launch_emu<k(), m(), i()>(ep, nunits, st);
    });
    return e;
}

cudaError_t prepare_emu_kernels() {
    cudaError_t e = cudaSuccess;
    emu::for_each_emu([&](auto k, auto m, auto i) {
        if (e == cudaSuccess) e = emu::ensure_emu_attr<k(), m(), i()>();
    });
    return e;
}

// whether a pass of this kind can hand over integers: |T'| < 2^60
bool emu_hands_over(int kind) {
    PassParams<double> p;
    std::memset(&p, 0, sizeof p);
    fill_taps(p, kind, 1.0);
    emu::Sched s;
    return emu::build_sched(kind, p, s) && s.tbits <= 60;
}

namespace emu {
// An mbarrier that nothing arrives on, waited for with a bound of `cycles`:
// the expiry path of the bounded waits, exercised without a fault.
__global__ void wait_probe_kernel(long long cycles) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(su32(&bar)), "r"(1));
    const long long t0 = clock64();
    while (true) {
        uint32_t ok;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     "selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok) : "r"(su32(&bar)), "r"(0u) : "memory");
        if (ok) return;
        if (clock64() - t0 > cycles) {
            atomicAdd(&g_emu_timeouts, 1u);
            return;
        }
    }
}
}  // namespace emu

cudaError_t emu_wait_probe(double ms, cudaStream_t st) {
    int dev = 0, khz = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev) != cudaSuccess || khz <= 0)
        khz = 2000000;   // SM clock unknown: assume 2 GHz
    const long long cycles = (long long)(ms * (double)khz);
    emu::wait_probe_kernel<<<1, 32, 0, st>>>(cycles);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t emu_take_timeouts(unsigned* count) {
    unsigned v = 0, z = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_emu_timeouts, sizeof v);
    if (e != cudaSuccess) return e;
    if (v) e = cudaMemcpyToSymbol(g_emu_timeouts, &z, sizeof z);
    *count = v;
    return e;
}

}  // namespace wvl
