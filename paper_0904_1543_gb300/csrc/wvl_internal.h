// Internal declarations shared by the host API and the kernel translation
// units.  Not part of the public ABI (see include/wvl.h).
#pragma once
#include <cstddef>
#include <cstdint>

#include <cuda_runtime_api.h>

#include "wvl.h"

namespace wvl {

// Filters of the method, derived on the host (filters.cpp).
struct FilterSet {
    double h[16];   // h_j, j = -7..8         (Eq. refinement)
    double g[16];   // g_j = (-1)^j h_{1-j}
    double w[16];   // w_k, k = k0..k0+15     (Eq. magicfilter)
    double a[29];   // a_l, l = -14..14       (Eqs. kiner, fprod)
    int k0;
};
const FilterSet& filters();

// The five 1D operators.  Each 3D operator is three passes of
// F(I, a) = sum_t f_t G(a, I - HL + off + t), output written transposed
// (Eqs. 1dconvtrans and kinetic1d).
enum Kind { K_SYN = 0, K_ANA = 1, K_MF = 2, K_MFT = 3, K_KIN = 4, NKIND = 5 };

// Load/epilogue variants of a pass.
enum Mode {
    M_PLAIN = 0,   // read lines, write transposed
    M_UNCOMP = 1,  // synthesis pass 1: gather lines from the compressed layout
    M_COMP = 2,    // analysis pass 3: scatter into the compressed layout
    M_POT = 3,     // magic-filter pass 3: V*psi, rho += occ psi^2, Epot partials
    M_KMID = 4,    // kinetic pass 1/2: K_p = T*G + K_{p-1}, G_p = G^T
    M_KLAST = 5,   // kinetic pass 3: K_3 and sum s*(K_3 - K0) partials
    NMODE = 6
};

constexpr int MAXSEG = 8;      // cells (segments) per launch
constexpr int NTHREADS = 128;  // threads per CTA (4 warps)
// register-resident density outputs per thread in the FP64 M_POT pass (the
// FP32 pass, pass32.cu, keeps its compensated density sums in shared memory)
constexpr int POT_OUT = 32;
constexpr int MAX_FINE = 1024; // largest fine extent of one axis

// One cell's orbitals inside one pass launch.  Element offsets are per
// orbital; orbital o of the segment starts at o * P in every array (P = fine
// points = compressed length).
template <typename T>
struct Seg {
    const T* in;          // pass input (orbital 0 of the segment)
    T* out;               // pass output (may be null for reduction-only M_POT/M_KLAST)
    const T* in2;         // K_{p-1} for M_KMID/M_KLAST (null = 0)
    T* out2;              // G_p for M_KMID
    const T* aux;         // M_POT: V (null = no potential);  M_KLAST: K0 (null = 0)
    double* rho;          // M_POT: density target (null = none)
    double* part;         // per (orbital, tile) partial sums, [norb][tiles]
    const double* occ;    // M_POT: occupations of the segment's orbitals
    const double* gscale; // M_COMP: when set, output o is scaled by 2 occ[o] gscale[0]
                          //   (dE_loc/dpsi = 2 occ g H psi, the adjoint of E_loc)
    const double* eps;    // M_KMID pass 1 without in2: K_0 = -eps[o] G (Helmholtz shift)
    const int* mapc;      // M_UNCOMP/M_COMP with a localisation region: coarse point ->
    const int* mapf;      //   position of c^0 / index k of c^{1..7} (ncoarse + 7k), or -1
    const int* lexp;      // emulated M_UNCOMP: largest biased exponent of each input line,
                          //   [orbital][line] (null: the pass scans its lines)
    const int* gin;       // emulated passes: the input is integers, element e of scale
    const int* gmax;      //   2^gin[orbital][e mod nsrc] (null: FP64); gmax[orbital][slot][line]:
                          //   exponents of each line's largest (emu::hand_slots)
    int* gout;            // the output is integers, line a's of scale 2^gout[orbital][a], and
    int* gtop;            //   gtop is gmax of the pass that reads them, on lines of nnext
    int nsrc, nnext;
    long long clen;       // compressed length of one orbital (orbital stride there)
    long long ncoarse;    // scaling coefficients stored (start of the wavelet block)
    int bx1, bx2, bx3;    // free/surface boundary conditions: box extents inside the
    int bo1, bo2, bo3;    //   padded cell and its offsets (coarse points); bx1 = 0 otherwise
    int nin;              // free lines (no wrap; 0 = periodic lines): input line length;
    int inoff;            //   row slot j holds input element j - hl + inoff, zero outside
    long long Pin;        //   [0, nin); Pin = input elements per orbital
    int vN1, vN2, vN3;    // M_POT on free lines: V and rho live on another grid (extents
    int vo1, vo2, vo3;    //   vN1, vN2, vN3, vP elements); output (X1, X2, I) sits there at
    long long vP;         //   (X1 + vo1, X2 + vo2, I + vo3) modulo the extents; vN1 = 0: same
                          //   layout as the output
    int go1, go2, go3;    // free lines over a region's box: the box origin in the cell and
    int gc1, gc2, gc3;    //   the cell's coarse extents (region index lookups, with wrap);
                          //   gc1 = 0 otherwise
    long long P;          // elements per orbital
    long long rho_gstride;// M_POT: 0 -> rho += (direct), else group g writes rho[g*stride]
    long long blk0;       // first work unit of the segment in the launch
    int n, N;             // line length and line count of this pass
    int N1, N2;           // fine extents (index decoding)
    int n1, n2;           // coarse extents (compressed layout)
    int norb;
    int tiles;            // work units per orbital (group): ceil(N / LT), times nwin when emulated
    int nwin;             // emulated FP64 passes: output windows per line
    int opg;              // M_POT: orbitals per group
    int rowlen;           // shared-memory row length in elements
};

// A work unit is one (orbital, tile) -- or, for M_POT, one (orbital group,
// tile) whose orbitals the CTA walks in order.  The kernel is persistent:
// CTA b takes units b, b + gridDim.x, ... and stages the next job in the
// second shared-memory buffer while it computes the current one.
template <typename T>
struct PassParams {
    T f[2][32];           // taps per output parity (single-parity kinds: both equal)
    float2 tp[32];        // FP32: tap pairs of outputs 2m, 2m + 1 (pass_kernel.cuh)
    long long nunits;     // work units over all segments
    int bufelems;         // elements of one staging buffer (two are allocated)
    int hl;               // left halo
    int LT;               // lines per tile (power of two, 4..32)
    int nseg;
    Seg<T> seg[MAXSEG];
};

// ------------------------------------------------ fused plane/column chain
// The local Hamiltonian chain as five kernels (fused_kernel.cu): each xy plane
// kernel keeps one fine-grid plane of an orbital in shared memory and applies
// the axis-1 and axis-2 filters of one or more operators to it; each column
// kernel keeps N3 x 32-column (FP64: 16) tiles and applies the axis-3
// filters.  Programs, in chain order (a = S3 c, s = S1 S2 a):
enum FzProg {
    FZ_SYN3 = 0,    // column: gather c from the compressed form, a = S3 c
    FZ_SKM12 = 1,   // plane:  s = S1 S2 a;  v = (T1 + T2) s (Ekin part);  t = MF1 MF2 s
    FZ_POT3 = 2,    // column: psi_r = MF3 t;  V psi_r, rho, Epot;  x = MFT3 (V psi_r)
    FZ_MFTA12 = 3,  // plane:  w' = A1 A2 (MFT1 MFT2 x + v)
    FZ_TA3 = 4,     // column, two I2 rows: H psi = A3 (w' + T3 a) (Ekin part), compressed
    FZ_NPROG = 5
};
constexpr int FZ_PTHREADS = 512;   // plane kernels: most threads (fz_plane_shape)
constexpr int FZ_CTHREADS = 128;   // column kernels
constexpr int FZ_RR = 8;           // row-pass outputs per thread (along the row)
constexpr int FZ_RC = 8;           // column-pass outputs per thread (along the column)
constexpr int FZ_MIN_FINE = 32;    // fine extents the fused chain takes: multiples
constexpr int FZ_MAX_FINE = 128;   //   of 8 in [32, 128]
constexpr int FZ_EPW = 64;         // FZ_POT3: orbitals whose Epot partials are held at once
template <typename T>
__host__ __device__ constexpr int fz_ltc() { return 128 / (int)sizeof(T); }   // tile columns

template <typename T>
struct FzSeg {
    const T* in;          // program input (FZ_SYN3: compressed psi)
    const T* in2;         // FZ_MFTA12: v;  FZ_TA3: a
    T* out;               // program output (FZ_TA3: compressed H psi)
    T* out2;              // FZ_SKM12: v
    T* out3;              // FZ_SKM12: t
    const T* V;           // FZ_POT3: potential
    double* rho;          // FZ_POT3: density target (null = none)
    long long rho_gstride;// 0 -> rho += ; else group g writes rho[g * stride]
    const double* occ;    // FZ_POT3: occupations;  FZ_TA3 with gscale: the scale's occ
    const double* gscale; // FZ_TA3: when set, H psi of orbital o is scaled by 2 occ[o] gscale[0]
    double* part;         // energy partials [norb][ptiles]; this program writes from poff
    long long P;          // fine points per orbital
    long long blk0;       // first job of the segment in the launch
    int N1, N2, N3, n1, n2;
    int norb, opg;        // FZ_POT3: orbitals per group
    int ncb;              // column blocks per row, ceil(N1 / fz_ltc)
    int ptiles, poff;
    int RS;               // shared-memory row stride in elements
};

// Launch shape of a plane kernel (fz_plane_shape): threads, register cap, and of the transposing
// form (fused_plane.cu) the side of its planes (0: the general form) and the CTAs per SM that
// walk over the planes (0: a CTA per plane).
struct FzShape {
    int threads = 0, regs = 0, rs = 0, ctas = 0;
    bool operator!=(const FzShape& o) const {
        return threads != o.threads || regs != o.regs || rs != o.rs || ctas != o.ctas;
    }
};

template <typename T>
struct FzParams {
    T tap[4][2][32];      // the program's filters, per output parity (see fused_kernel.cu)
    float2 tp[4][32];     // FP32 row passes: tap pairs of outputs 2m, 2m + 1 (fused_kernel.cu)
    long long njobs;
    FzShape shape;        // plane kernels: one launch shape per launch
    int nseg;
    FzSeg<T> seg[MAXSEG];
};

// Parameters of the transposing plane kernels: every tap twice (packed FMAs on two lines)
struct FzTileParams {
    float2 td[4][2][32];
    float2 tp[2][32];     // the row filters' tap pairs of outputs 2m, 2m + 1
    long long njobs;
    int nseg;
    FzSeg<float> seg[MAXSEG];
};
// the launch shape of a program on planes of N1 x N2 (rs = 0: not taken)
FzShape fz_tplane_shape(int prog, int N1, int N2);
cudaError_t launch_tplane(int prog, const FzParams<float>& p, cudaStream_t st);
cudaError_t prepare_tplane(int prog, FzShape s);

// shared-memory row stride of an xy plane with N1 columns: a 16-byte multiple
// whose count of 16-byte words is odd (lane-per-row vector loads hit distinct banks)
template <typename T>
inline int fz_plane_rs(int N1) {
    const int v = 16 / (int)sizeof(T);
    int w = (N1 + v - 1) / v;
    if ((w & 1) == 0) ++w;
    return w * v;
}
// Square FP32 planes of 32 to 128 points a side in steps of 32 take the transposing form
// (fused_plane.cu, with both sides measured).  The others: threads of a plane kernel, by the
// CTAs whose two planes fit in an SM's shared memory and by the column items of a plane (8 rows
// of a 16-byte column; a last round of few items wastes the CTA); registers as compiled, or
// capped at 96 where that lets one more CTA in.  More planes per SM overlap one's loads and
// barriers with another's filters.  FP32, microseconds per call of 2560 planes of 40 (of 640, one
// figure each, for SYN3 + SKM12 / MFTA12), with 256 threads and as chosen:
//   one CTA       512: 120^2 404 / 212 and 378 / 186
//   two, three    256 (80x88, 220 items: 177 / 75, with 160 185 / 84).  SKM12 160 where three
//                 CTAs fit (256 threads leave registers for two), 256 would leave a second
//                 round of at most 64 items, and rows are chunks of 8 (N1 no multiple of
//                 16: twice the row items, which hide the fewer threads): 104x88, 286 items,
//                 237 and 228; 88x96 218 and 203; 120x72 231 and 221; but 112x80 228 and 232,
//                 88x112 (two CTAs) 255 and 289, and 480 planes of 104x88, two waves either
//                 way, 64 and 72
//   four          SKM12 128: 80^2 170 and 160; MFTA12 256
//   five to seven 128 at 96 registers / 160: 72^2 174 / 67 and 154 / 63, 64x80 145 / 62 and
//                 130 / 56
//   eight, nine   128 at 96 / 128: 72x40 118 / 47 and 100 / 39, 56^2 113 / 46 and 99 / 40
//   more          MFTA12 96: 48^2 43 and 33, 40^2 39 and 29; SKM12 at 96 registers 96 for 65 to
//                 83 items, 48^2 92 and 77; 64 for fewer, 40^2 100 and 74 (96: 79); one
//                 warp for planes of one warp's items
// Launches of at most two planes per SM keep 256 threads, SKM12 at four CTAs and MFTA12 of at most
// three (six for planes of one warp's items): there a plane's own time counts (320 planes of
// 72^2: MFTA12 16.5 with 256, 18.5 with 160; of 32^2 9.7 and 12.3).  FP64
// planes are bound by the FP64 pipe.  regs: 0 as compiled, else the cap.
template <typename T>
inline FzShape fz_plane_shape(int prog, int N1, int N2, long long planes) {
    if (sizeof(T) == 8 || planes <= 2 * 152) return {256, 0};
    const FzShape ts = fz_tplane_shape(prog, N1, N2);
    if (ts.rs > 0) return ts;
    // (static and reserved shared memory: 1792 bytes of the SM's 228 KB per CTA)
    const int smem = 2 * N2 * fz_plane_rs<T>(N1) * (int)sizeof(T) + 1792;
    const int ctas = 228 * 1024 / smem;
    const int items = (N2 / FZ_RC) * (N1 * (int)sizeof(T) / 16);
    if (ctas <= 1) return {512, 0};
    if (prog == FZ_MFTA12) {
        if (ctas <= 4 || planes <= (items <= 32 ? 6 : 3) * 152) return {256, 0};
        return {items <= 32 ? 32 : ctas <= 7 ? 160 : ctas <= 9 ? 128 : 96, 0};
    }
    if (ctas == 2) return {256, 0};
    if (ctas == 3) {
        const bool fewer = (planes + 455) / 456 < (planes + 303) / 304;   // waves of three and of two
        return {fewer && items > 256 && items <= 320 && N1 % 16 != 0 ? 160 : 256, 0};
    }
    if (ctas == 4) return {planes <= 3 * 152 ? 256 : 128, 0};
    return {items <= 32 ? 32 : items <= 64 ? 64 : items < 84 ? 96 : 128, 96};
}
template <typename T>
size_t fz_smem(int prog, int N1, int N2, int N3);
template <typename T>
cudaError_t launch_fused(int prog, const FzParams<T>& p, size_t smem, cudaStream_t st);
template <typename T>
cudaError_t prepare_fused_kernels();

// Per-kind geometry: taps, parity offsets, left/right halo.
struct KindGeom {
    int nt, off0, off1, extra, hl, hr;
};
KindGeom kind_geom(int kind);

// Fills p.f and p.hl for a kind and axis spacing (kinetic only).
template <typename T>
void fill_taps(PassParams<T>& p, int kind, double hgrid);

// Launches one pass.  R (outputs per thread) must be 4 or 8.
template <typename T>
cudaError_t launch_pass(int kind, int mode, int R, const PassParams<T>& p,
                        long long nunits, size_t smem, cudaStream_t st, bool persistent);

// The FP32 passes of pass32.cu: threads and shared memory of a launch whose longest
// output line is n (rho: the potential pass has density sums), and the launch.
int pass32_threads(int LT, int nmax);
int pass32_ctas(int threads, size_t smem);   // potential pass: CTAs per SM
size_t pass32_smem(int kind, int mode, int LT, int n, bool rho);
cudaError_t launch_pass32(int kind, int mode, const PassParams<float>& p, long long nunits, int threads,
                          size_t smem, cudaStream_t st);
cudaError_t prepare_pass32();

// Sets the dynamic shared-memory attribute of every pass kernel on the
// current device (done lazily by launch_pass too; needed before capture).
template <typename T>
cudaError_t prepare_pass_kernels();

// Preconditioned conjugate gradient on compressed coefficients (pcg.cu).
struct PcgParams {
    double diag[8];       // diagonal of S^T K S per component mu
    const double* eps;    // per-orbital shift (device)
    double* part;         // block partials [norb][nblk]
    long long len;        // compressed length per orbital (8 m)
    long long m;          // coarse points
    int norb;
    int nblk;             // blocks per orbital
};
enum PcgOp { PCG_INIT = 0, PCG_DOT = 1, PCG_STEP = 2, PCG_DIR = 3 };
// INIT: (a=x, b=r, c=z, d=p, e=g);  DOT: (a, b) -> partials;
// STEP: (a=x, b=r, c=z, d=p, e=Ap, s1=rz, s2=pq);  DIR: (a=p, c=z, s1=rz_new, s2=rz_old)
template <typename T>
cudaError_t launch_pcg(int which, const PcgParams& q, T* a, T* b, T* c, T* d, const T* e,
                       const double* s1, const double* s2, cudaStream_t st);

// The preconditioner in FP32 by the separable operator (helmholtz.cu), ncg >= 1
// iterations: buf = five arrays of norb P floats, scal = three of norb doubles, part =
// partials of norb x 64 and of norb x ceil(N1 N2 / 32) doubles.
bool helmholtz_pcg_ok(const int Nf[3], int norb);
cudaError_t launch_helmholtz_pcg(const int Nf[3], const double hg[3], const double diag[8], int norb,
                                 const float* g, const double* eps, int ncg, float* x, double* rr,
                                 float* const buf[5], double* const scal[3], double* const part[2],
                                 cudaStream_t st);

// Kernel-launch counter behind wvl_kernel_launches().
void count_launches(unsigned long long k);
// Status with a detail string for wvl_last_error() (thread-local), and its reset.
wvl_status set_error(wvl_status s, const char* msg);
void clear_error();

// ekin/epot finalisation and density reduction.
cudaError_t launch_reduce_parts(const double* part, const double* minus, int tiles,
                                int norb, double* out, cudaStream_t st);
cudaError_t launch_rho_reduce(const double* parts, long long P, int ngroups,
                              double* rho, cudaStream_t st);
// several reduce_parts sums in one launch: task k covers warps
// warp0 .. warp0 + norb - 1, out[o] = sum part[o][*] - sum mpart[o][*]
struct PartTask {
    const double* part;
    const double* mpart;  // null: nothing subtracted
    double* out;
    int tiles, mtiles, norb, warp0;
};
constexpr int MAXTASK = 2 * MAXSEG;
struct PartTasks {
    PartTask t[MAXTASK];
    int ntask = 0;
    int nwarps = 0;
    // append a task; false when the table is full
    bool add(const double* part, int tiles, const double* mpart, int mtiles, double* out, int norb) {
        if (ntask >= MAXTASK) return false;
        t[ntask] = PartTask{part, mpart, out, tiles, mtiles, norb, nwarps};
        ++ntask;
        nwarps += norb;
        return true;
    }
};
cudaError_t launch_reduce_parts_multi(const PartTasks& t, cudaStream_t st);
// scalar products on the tensor cores (overlap_mma.cu): workspace bytes and launch;
// bounded waits that ran out since the last call are added to *count
size_t overlap_mma_ws(int na, int nb, long long len, bool sym);
size_t overlap_mma_ws_bound(int na, int nb, long long len);   // of every call of at most these sizes
cudaError_t launch_overlap_mma(int prec, int na, const void* a, int nb, const void* b, long long len,
                               bool sym, double* S, void* ws, cudaStream_t st);
cudaError_t overlap_take_timeouts(unsigned* count);
// E_loc = sum_o occ (ekin + epot) into *out (one fixed-order CTA), and
// dV = gbar rho in the potential's precision (the adjoint of E_loc in V).
cudaError_t launch_eloc_total(const double* occ, const double* ekin, const double* epot,
                              int norb, double* out, cudaStream_t st);
template <typename T>
cudaError_t launch_scale_density(const double* rho, const double* gbar, long long P, T* dV,
                                 cudaStream_t st);

}  // namespace wvl
