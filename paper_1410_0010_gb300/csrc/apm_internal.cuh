// apm_internal.cuh -- device descriptors and kernel entry points shared by the
// translation units of libapm (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "apm.h"

namespace apm {

// ---------------------------------------------------------------------------
// compile-time sizes
// ---------------------------------------------------------------------------
constexpr int kMaxStages = 12;      // radix stages of one 1-D transform
constexpr int kFftThreads = 256;    // most threads of an FFT pass CTA (launch bound)
// complex elements one buffer of a pass CTA aims at by default (lines x length)
constexpr int kFftBudgetF32 = 2048;
constexpr int kFftBudgetF64 = 1024;
constexpr int kFftSmemLimit = 200 * 1024;   // dynamic shared memory a pass CTA may take

// the five FFT passes of a level solve
enum { kPassXf = 0, kPassYf = 1, kPassZ = 2, kPassYi = 3, kPassXi = 4, kFftPasses = 5 };

inline int pow2_floor_i(int v) {
    int p = 1;
    while (p * 2 <= v) p *= 2;
    return p;
}
// lines per CTA of a pass for a transform of length L and a buffer budget (in
// complex elements): a power of two; row pairs 1..32 for the x passes, kx
// columns 4..32 (FP64 2..32) for the y/z passes (at least 32 contiguous bytes
// of each row a line group reads)
inline int fft_pass_lines(int pass, int L, int budget, bool f64) {
    const int v = pow2_floor_i(std::max(1, budget / L));
    if (pass == kPassXf || pass == kPassXi) return std::min(32, v);
    return std::min(32, std::max(f64 ? 2 : 4, v));
}
// bytes of the x-forward pass's int64 row staging area (2 lines rows of G0
// cells, rounded to 128 bytes) plus its mbarrier
__host__ __device__ inline size_t fft_xf_stage_bytes(int lines, int G0) {
    return ((size_t)2 * lines * G0 * 8 + 127) / 128 * 128 + 128;
}
// dynamic shared memory of a pass CTA: two buffers plus the twiddles (the x
// passes pad each element row to lines + 1); the x-forward pass also stages
// its GMF rows (G0: the GMF row length)
inline size_t fft_pass_smem(int pass, int L, int lines, size_t csz, int G0 = 0) {
    if (pass == kPassXf) return (size_t)(2 * L * (lines + 1) + L) * csz + fft_xf_stage_bytes(lines, G0);
    if (pass == kPassXi) return (size_t)(2 * L * (lines + 1) + L) * csz;
    return (size_t)(2 * L * lines + L) * csz;
}
constexpr int kMaxFft = 1024;       // longest supported transform

// device status bits (latched with atomicOr, read by apm_sync_status)
constexpr unsigned kStOverflow = 1u;
constexpr unsigned kStOutOfBox = 2u;
constexpr unsigned kStTimeout = 4u;
constexpr unsigned kStBounds = 8u;

// Bounds-checked builds (-DAPM_BOUNDS_CHECK): the kernels test each global
// index whose value depends on the data or the hierarchy before using it; an
// index outside [0, n) sets the status word's bounds bit (apm_sync_status:
// APM_E_BOUNDS) and the access is skipped.  Release builds compile the tests
// out.  Nothing here asserts or traps.
#ifdef APM_BOUNDS_CHECK
__device__ __forceinline__ bool in_bounds(long long i, long long n, unsigned* status) {
    if (i >= 0 && i < n) return true;
    if (status) atomicOr(status, kStBounds);
    return false;
}
#define APM_IN_BOUNDS(i, n, status) ::apm::in_bounds((long long)(i), (long long)(n), (status))
#else
#define APM_IN_BOUNDS(i, n, status) true
#endif

template <typename T> struct Cplx;
template <> struct Cplx<float> { using type = float2; };
template <> struct Cplx<double> { using type = double2; };

// One mixed-radix 1-D transform of length L (Stockham, radices in order).
struct FftPlan1D {
    int L;
    int nst;
    int tw_off;                       // offset of exp(-2 pi i t/L), t < L, in the twiddle arenas
    unsigned char radix[kMaxStages];
    // per stage: Ns (product of the radices before it), the twiddle stride
    // L / (Ns R), and ceil(2^32 / Ns) for exact division of small integers
    // (n < 2^21) by Ns as __umulhi(n, magic) (Ns = 1: magic 0, q = n)
    unsigned short ns[kMaxStages];
    unsigned short step[kMaxStages];
    unsigned magic[kMaxStages];
};

// Stage radices of a length-L transform: greedily the largest allowed radix
// (at most max_radix) that divides what is left.  Radices above 8 are
// composites of two of 2, 3, 4, 5, 7, 8 run in registers (FP32 path only).
inline bool fft_plan(int L, int max_radix, FftPlan1D* pl) {
    static const int kSimple[] = {8, 7, 5, 4, 3, 2};
    static const int kWithComposite[] = {16, 15, 14, 12, 10, 9, 8, 7, 6, 5, 4, 3, 2};
    pl->L = L;
    pl->nst = 0;
    if (L < 2) return false;
    int n = L;
    while (n > 1) {
        int pick = 0;
        if (max_radix <= 8) {
            for (int r : kSimple)
                if (n % r == 0) { pick = r; break; }
        } else {
            for (int r : kWithComposite)
                if (r <= max_radix && n % r == 0) { pick = r; break; }
        }
        if (!pick || pl->nst >= kMaxStages) return false;
        pl->radix[pl->nst++] = (unsigned char)pick;
        n /= pick;
    }
    int Ns = 1;
    for (int st = 0; st < pl->nst; ++st) {
        pl->ns[st] = (unsigned short)Ns;
        pl->step[st] = (unsigned short)(L / (Ns * pl->radix[st]));
        pl->magic[st] = Ns == 1 ? 0u : (unsigned)((0x100000000ULL + Ns - 1) / Ns);
        Ns *= pl->radix[st];
    }
    return true;
}

// The same transform with the radices in reverse order (the inverse column
// transforms: the z pass's inverse starts with the radix its forward ends on).
inline void fft_plan_reversed(const FftPlan1D& f, FftPlan1D* r) {
    *r = f;
    for (int st = 0; st < f.nst; ++st) r->radix[st] = f.radix[f.nst - 1 - st];
    int Ns = 1;
    for (int st = 0; st < r->nst; ++st) {
        r->ns[st] = (unsigned short)Ns;
        r->step[st] = (unsigned short)(r->L / (Ns * r->radix[st]));
        r->magic[st] = Ns == 1 ? 0u : (unsigned)((0x100000000ULL + Ns - 1) / Ns);
        Ns *= r->radix[st];
    }
}

// ---- transforms with compile-time plans (fft_fast.cuh) -----------------------
// Lengths with a compile-time radix plan: X(L, R1, R2, R3); R3 = 1 for two
// stages.  Every radix is one the butterflies compute in registers.  They
// cover every {2,3,5,7}-smooth length from 36 to 150 (a refined grid of N cells
// takes the smallest one >= N + 20; an isolated root of N cells takes 2 N) and
// the usual longer ones; the rest runs the runtime-planned kernels.  The lists
// are four groups so that they compile in parallel.  FP64 takes groups 1 to 3:
// below 70 points it runs the runtime-planned kernels, as it always has (no plan was
// measured there).
#define APM_FAST_LENGTHS_0(X) \
    X(36, 6, 6, 1) X(40, 8, 5, 1) X(42, 7, 6, 1) X(45, 9, 5, 1) X(48, 8, 6, 1) X(49, 7, 7, 1) \
    X(50, 10, 5, 1) X(54, 9, 6, 1) X(56, 8, 7, 1) X(60, 10, 6, 1) X(63, 9, 7, 1) X(64, 8, 8, 1)
#define APM_FAST_LENGTHS_1(X) \
    X(70, 10, 7, 1) X(72, 9, 8, 1) X(75, 15, 5, 1) X(80, 10, 8, 1) X(81, 9, 9, 1) X(84, 12, 7, 1) \
    X(90, 10, 9, 1) X(96, 12, 8, 1) X(98, 14, 7, 1) X(100, 10, 10, 1) X(105, 15, 7, 1) X(108, 12, 9, 1)
#define APM_FAST_LENGTHS_2(X) \
    X(112, 14, 8, 1) X(120, 12, 10, 1) X(125, 5, 5, 5) X(126, 14, 9, 1) X(128, 16, 8, 1) X(135, 15, 9, 1) \
    X(140, 14, 10, 1) X(144, 12, 12, 1) X(147, 7, 7, 3) X(150, 15, 10, 1)
#define APM_FAST_LENGTHS_3(X) \
    X(160, 16, 10, 1) X(168, 14, 12, 1) X(180, 15, 12, 1) X(192, 16, 12, 1) X(200, 10, 5, 4) X(216, 6, 6, 6) \
    X(224, 16, 14, 1) X(240, 16, 15, 1) X(250, 10, 5, 5) X(256, 16, 16, 1) X(288, 8, 6, 6) X(300, 10, 6, 5) \
    X(320, 8, 8, 5) X(360, 10, 6, 6) X(384, 8, 8, 6) X(400, 10, 8, 5) X(480, 10, 8, 6) X(512, 8, 8, 8)
constexpr int kFastGroups = 4;
// lines per CTA: kx columns of a column pass, complex lines (row pairs) of an
// x pass; 128 bytes of each HBM row in both precisions
constexpr int fast_lines(bool f64) { return f64 ? 8 : 16; }

// threads of a fast pass CTA for `lines` lines: whole warps.  Up to L = 96, of 3
// to 6 warps the count whose stages leave the fewest threads without a butterfly
// in their last trip; above, 4 or, where that fits the first stage's butterflies,
// 5; FP32 above 192 8, FP64 there as many as give 24 warps per SM (its pipe
// bounds it: up to 320 it takes the same time with 4 to 8).  The z pass of 32
// grids of L = 150: 264 us with 2 warps, 178 with 3, 181 with 4, 171 with 5; 8
// spectral ones of 120: 155 with 3, 131 with 4; 343 grids of 36 to 84: all passes
// 531 with 2 or more, 498 with 3 or more, 515 with 3 always.  A periodic root's
// five passes with 4, 6 and 8 warps: 200^3 147, 139, 129 us; 240^3 228, 242, 196;
// 256^3 251, 253, 215; 320^3 549, 497, 460; 512^3 2133, 1879, 1692.
constexpr int fast_threads(int r1, int r2, int r3, int lines) {
    const int L = r1 * r2 * r3;
    const int items[3] = {L / r1 * lines, L / r2 * lines, r3 > 1 ? L / r3 * lines : 0};
    if (L > 192 && lines == 16) return 256;
    if (L > 96) {
        const int ctas = 220 * 1024 / (L * 17 * 8);   // per SM, by their shared memory
        int nt = items[0] > 128 && items[0] <= 160 ? 160 : 128;
        while (nt < 256 && nt * ctas < 768) nt += 32;
        return nt;
    }
    int best = 96, best_cost = 1 << 30;
    for (int nt = 96; nt <= 192; nt += 32) {
        int cost = 0;
        for (int k = 0; k < 3; ++k) cost += (items[k] + nt - 1) / nt * nt;
        if (cost < best_cost || (cost == best_cost && nt <= 160)) {
            best = nt;
            best_cost = cost;
        }
    }
    return best;
}
// the group of length L's compile-time plan, -1 without one
inline int fast_group(int L, bool f64) {
#define APM_FAST_CASE(LL, A, B, C) if (L == LL) return g;
    int g = 0;
    if (!f64) { APM_FAST_LENGTHS_0(APM_FAST_CASE) }
    g = 1;
    APM_FAST_LENGTHS_1(APM_FAST_CASE)
    g = 2;
    APM_FAST_LENGTHS_2(APM_FAST_CASE)
    g = 3;
    APM_FAST_LENGTHS_3(APM_FAST_CASE)
#undef APM_FAST_CASE
    return -1;
}
inline bool fast_length(int L, bool f64) { return fast_group(L, f64) >= 0; }
constexpr size_t fast_csz(bool f64) { return f64 ? sizeof(double2) : sizeof(float2); }
// dynamic shared memory of a fast column-pass CTA: the buffer and the twiddles
constexpr size_t fast_col_smem(int L, bool f64) { return (size_t)(L * fast_lines(f64) + L) * fast_csz(f64); }
// ... and of a fast x-pass CTA (rows padded to one line more; the x-inverse
// pads its lines by one element every R_last positions: at most L / 2 more)
constexpr size_t fast_row_smem(int L, bool f64) {
    return (size_t)(L * (fast_lines(f64) + 1) + L / 2 + L) * fast_csz(f64);
}

// Column-pass chunks carry (kx tile, line index of the other axis) as
// (kt << 20) | other: other < 2^20, kt < 2^11.
constexpr int kColOtherBits = 20;

// Everything a kernel needs to know about one grid.
struct GridDev {
    int kind;            // Green's table: 0 refined, 1 periodic root, 2 isolated root
    int mode;            // deposit edge rule: 0 drop, 1 fold, 2 wrap
    int N[3];            // interior cells
    int G[3];            // GMF box
    int M[3];            // FFT lengths
    int W[3];            // window N + 4 (cells [-2, N+2))
    int s0[3];           // M index of window cell -2, in [0, M)
    int Hx;              // M[0]/2 + 1 (half spectrum along x)
    int Hy2, Hz2;        // M[1]/2 + 1, M[2]/2 + 1 (octant table)
    long long lo[3];     // global level index of GMF cell 0
    long long start[3];  // global level index of interior cell 0
    int parent;          // index of the parent among the grids of level - 1, or -1
    int pN[3];
    long long pstart[3];
    double delta;
    FftPlan1D fx, fy, fz;
    FftPlan1D iy, iz;    // fy, fz with the radices reversed (inverse column transforms)
    long long tab_off;   // octant table offset (elements) in the table arenas
    long long wsA, wsB;  // workspace offsets (complex elements)
    long long cells_gmf; // G0 G1 G2
    int lines[kFftPasses];   // lines per CTA of each pass (row pairs for xf / xi)
    int rows_gas;        // GMF rows per CTA of the baryon initialisation
    int acc_sh[3];       // 1 when output cell 0 is the second cell of its block, else 0
    int acc_nb[3];       // output blocks per axis
    double inv2d;        // 1 / (2 delta)
    double inv_m3;       // 1 / (M0 M1 M2), the inverse transform's normalisation
    int grad;            // gradient operator (apm_gradient): 0 two-point, 1 four-point, 2 spectral
    int h;               // phi_short window half-width: cells [-h, N+h) (3 four-point, else 2)
    double dk[3];        // 2 pi / (M_j delta): the spectral gradient's k per mode index
    double inv12d;       // 1 / (12 delta)
};

// Threads of a CTA walking a batch of rows [r0, r1) of length n in row-major
// order: thread t starts at element t and strides by the block size, the
// (row, x) pair stepped incrementally (no division per element).
struct RowWalk {
    int r, x, dr, dx, n;
    __device__ RowWalk(int r0, int n_) : n(n_) {
        r = r0;
        x = threadIdx.x;
        while (x >= n) {
            x -= n;
            ++r;
        }
        dr = blockDim.x / n;
        dx = blockDim.x - dr * n;
    }
    __device__ void next() {
        x += dx;
        r += dr;
        if (x >= n) {
            x -= n;
            ++r;
        }
    }
};

// 2x2x2 output blocks per CTA of the four-point acceleration kernel (flat ranges
// of the grid's blocks, x fastest, so every thread gets the same count)
constexpr int kAccBlocksPerCta = 512;
// threads of an acceleration CTA; the two-point and spectral kernels give each
// one (x, y) column of blocks and march through up to kAccMarch blocks of it (4
// to 16 measure alike on large levels; the host halves it while a level would
// leave SMs idle)
#ifndef APM_ACC_THREADS
#define APM_ACC_THREADS 128
#endif
constexpr int kAccThreads = APM_ACC_THREADS;
#ifndef APM_ACC_MARCH
#define APM_ACC_MARCH 8
#endif
constexpr int kAccMarch = APM_ACC_MARCH;

// Threads of a CTA walking the flat range [f0, f0 + count) of elements of rows
// of length n: thread t starts at f0 + t and strides by the block size, with
// (row, x) stepped incrementally (one division per thread).
struct FlatWalk {
    int r, x, dr, dx, n, left;
    __device__ FlatWalk(long long f0, int count, int n_) : n(n_) {
        const long long f = f0 + threadIdx.x;
        r = (int)(f / n);
        x = (int)(f - (long long)r * n);
        left = count - (int)threadIdx.x;
        dr = blockDim.x / n;
        dx = blockDim.x - dr * n;
    }
    __device__ bool ok() const { return left > 0; }
    __device__ void next() {
        left -= blockDim.x;
        x += dx;
        r += dr;
        if (x >= n) {
            x -= n;
            ++r;
        }
    }
};

// Tile lookup: level cell -> candidate grids (CSR per tile).
struct TileMap {
    long long lo[3];
    int shift;
    int nt[3];
    const int* dep_off;   // grids whose GMF box, grown by one cell, meets the tile
    const int* dep_list;
    const int* own_off;   // grids whose interior meets the tile
    const int* own_list;
};

struct Chunk { int grid; int tile; };   // one CTA of a batched pass

// Per-level device view (passed by value to kernels).
struct LevelDev {
    int level;
    int n;                 // grids on the level
    int is_root;
    int refine;
    const GridDev* g;      // n descriptors
    TileMap map;
    double delta;
    double inv_delta;      // 1/delta
    double delta0;         // root cell: fixed-point positions count 2^-31 root cells
    double inv_delta0;
    int delta0_pow2;       // delta0 is a power of two: x/delta0 == x*inv_delta0 exactly
    int frac_bits;         // 31 - level: fraction bits of a position on this level
    long long span;        // N0 2^31: the box in fixed-point units
    double box;
    double root_cells;     // cells of the root
    int periodic;
    int overlap;           // a tile lists more than one deposit candidate
    int div_known;         // div_known() may divide by delta0 with inv_delta0
    int pos_exp;           // delta0 = 2^(31 - pos_exp) when delta0_pow2: X = rint(x 2^pos_exp)
    unsigned* status;      // the context's device status word (bounds-checked builds)
};

// Fixed-point TSC (shared by the deposit and the interpolation).  A drifted
// coordinate x becomes X = rint(x/delta0 2^31) once; on a level with P fraction
// bits the cell is X >> P and t = (X mod 2^P)/2^P; the weights of cells i-1, i,
// i+1 are (1-t)^2/2, 3/4 - (t-1/2)^2, t^2/2 as exact integers on the scale 2^63.
constexpr int kPosBits = 31;
constexpr unsigned long long kOne63 = 1ULL << 63;

// rint(x 2^K), ties to even, of a finite double with |x 2^K| < 2^62, from its
// exponent and significand with integer operations; kNoFixed for larger or
// non-finite values.
constexpr long long kNoFixed = (long long)(1ULL << 63);
__device__ __forceinline__ long long scaled_rint_bits(double x, int K) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF);
    if (e == 0x7FF) return kNoFixed;
    if (e == 0) return 0;   // zero or subnormal: far below one unit here
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL;
    const int sh = e - 1075 + K;   // |x 2^K| = m 2^sh
    unsigned long long r;
    if (sh >= 0) {
        if (sh >= 10) return kNoFixed;   // m 2^sh >= 2^62
        r = m << sh;
    } else if (sh < -54) {
        r = 0;
    } else {
        const int t = -sh;
        r = m >> t;
        const unsigned long long rem = m & ((1ULL << t) - 1);
        const unsigned long long half = 1ULL << (t - 1);
        if (rem > half || (rem == half && (r & 1))) ++r;
    }
    return (b >> 63) ? -(long long)r : (long long)r;
}
static __device__ __noinline__ long long scaled_rint_any(double x, int K) { return scaled_rint_bits(x, K); }
// The same, ok cleared in the place of kNoFixed (scaled_rint_small: and beyond
// its range, |x 2^K| < 2^51).  For |x 2^K| < 2^51 (every coordinate and mass of an
// ordinary problem) one FP64 addition rounds: x + 1.5 2^(52-K) lies where an FP64
// unit in the last place is 2^-K, so its significand holds rint(x 2^K), ties to
// even.  That is 16 clocks of the FP64 pipe for a warp, where the integer route
// takes about 40 instructions; BITS takes that one, for kernels the FP64 pipe
// bounds (the FP64 interpolation).
__device__ __forceinline__ long long scaled_rint_small(double x, int K, bool& ok) {
    const int e = (__double2hiint(x) >> 20) & 0x7FF;   // |x| < 2^(e - 1022)
    ok = e + K < 1073 && K > -900 && K < 1000;
    const int chi = ((1023 + 52 - K) << 20) | 0x80000;
    const double t = __dadd_rn(x, __hiloint2double(chi, 0));
    return __double_as_longlong(t) - ((long long)chi << 32);
}
template <bool BITS = false>
__device__ __forceinline__ long long scaled_rint(double x, int K, bool& ok) {
    if constexpr (!BITS) {
        const long long v = scaled_rint_small(x, K, ok);
        if (ok) return v;
    }
    const long long r = BITS ? scaled_rint_bits(x, K) : scaled_rint_any(x, K);
    ok = r != kNoFixed;
    return ok ? r : 0;
}

// RN(x / d) for a divisor known in advance: y = RN(1 / d), and two corrections
// with exact FMA residuals.  The first makes the quotient faithful, the second
// rounds it correctly (Markstein 1990; Cornea, Harrison and Tang 2002, for a
// divisor whose significand is not all ones: checked on the host, as is the
// range of d).  5 FP64 operations; x outside [2^-800, 2^800) takes the general
// division, 0 included.
__device__ __forceinline__ double div_known(double x, double d, double y, bool known) {
    const unsigned e = (unsigned)((__double2hiint(x) >> 20) & 0x7FF);
    if (!known || e - 223u >= 1600u) return __ddiv_rn(x, d);
    double q = __dmul_rn(x, y);
    q = __fma_rn(__fma_rn(-q, d, x), y, q);
    return __fma_rn(__fma_rn(-q, d, x), y, q);
}

// x' = x + v half_dt in FP64 (two rounded operations)
__device__ __forceinline__ double drift_raw(double x, double v, double half_dt) {
    return __dadd_rn(x, __dmul_rn(v, half_dt));
}

// X = rint(x'/delta0 2^31), canonical: modulo the box on a periodic domain; on
// an isolated domain a coordinate inside [0, box) that rounds onto the upper
// face stays in the last cell
template <bool BITS = false>
__device__ __forceinline__ long long fixed_position(double xd, const LevelDev& L) {
    // a coordinate 2^31 root cells or more from the origin (or NaN) saturates at
    // -+2^62: far outside every box
    long long X;
    bool ok;
    if (L.delta0_pow2) {
        X = scaled_rint<BITS>(xd, L.pos_exp, ok);
    } else {
        X = scaled_rint<BITS>(div_known(xd, L.delta0, L.inv_delta0, L.div_known != 0), 31, ok);
    }
    if (!ok) X = xd > 0.0 ? (1LL << 62) : -(1LL << 62);
    if (L.periodic) {
        if (X < 0 || X >= L.span) {
            X %= L.span;
            if (X < 0) X += L.span;
        }
    } else if (X >= L.span && xd >= 0.0 && xd < L.box) {
        X = L.span - 1;
    }
    return X;
}

__device__ __forceinline__ long long tsc_fixed(long long X, int P, unsigned long long w[3]) {
    const long long i = X >> P;
    const unsigned f = (unsigned)X & ((1u << P) - 1u);   // P <= 31
    unsigned S1 = (1u << P) - f;            // 2^P - f, at most 2^31
    const int up = 62 - 2 * P;
    w[2] = ((unsigned long long)f * f) << up;
    w[0] = ((unsigned long long)S1 * S1) << up;
    w[1] = kOne63 - w[0] - w[2];
    return i;
}

// (a b + 2^62) >> 63 for a, b < 2^63: product of two weights on the scale 2^63,
// rounded half up
__device__ __forceinline__ unsigned long long wmul63(unsigned long long a, unsigned long long b) {
    unsigned long long lo = a * b;
    unsigned long long hi = __umul64hi(a, b);
    unsigned long long lo2 = lo + (1ULL << 62);
    hi += (lo2 < lo) ? 1ULL : 0ULL;
    return (hi << 1) | (lo2 >> 63);
}

// ---- bulk asynchronous copies (TMA engine, no tensor map) and mbarriers ----
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// makes the initialised barrier visible to the asynchronous (TMA) proxy
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// global -> shared bulk copy of `bytes` (a multiple of 16; both addresses
// 16-byte aligned), completing on `bar`
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// one poll of phase `parity`; a thread may be suspended up to kWaitHintNs
// nanoseconds inside it
constexpr unsigned kWaitHintNs = 1000;
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(kWaitHintNs)
        : "memory");
    return ok != 0;
}
// waits for phase `parity` of `bar` at most `limit` polls (about a second in
// all); false when it ran out
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned parity, unsigned limit) {
    for (unsigned it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
constexpr unsigned kWaitPolls = 1u << 20;

// wmul63 for a < 2^32 and a 32-bit result (a weight is at most 1): with
// b = bh 2^32 + bl, (a b + 2^62) >> 63 equals (a bh + ((a bl) >> 32) + 2^30) >> 31
// (the low 32 bits of a bl cannot carry into the result)
__device__ __forceinline__ unsigned wmul63_32(unsigned a, unsigned long long b) {
    const unsigned long long hi = (unsigned long long)a * (unsigned)(b >> 32) + (1ULL << 30);
    return (unsigned)((hi + __umulhi(a, (unsigned)b)) >> 31);
}

struct Particles {
    long long n;
    const double *x, *y, *z, *vx, *vy, *vz, *m;
    const int* perm = nullptr;   // processing order (launch_order): slot i visits particle perm[i]
    unsigned stride = 0;         // the deposit's walk through its CTAs in that order (deposit_order)
    bool spread = false;         // ... and its lanes' slots (thread_slot)
    __device__ __forceinline__ long long at(long long i) const { return perm ? (long long)perm[i] : i; }
};

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
// Every kernel of a solve is launched as a programmatic dependent of the one
// before it on its stream, so the launch itself overlaps that one's end; each
// begins with begin_kernel(), which waits until everything before it is complete
// and visible (nothing is read or written early, whatever comes before: a kernel
// of the caller's, a copy, another stream joined by an event).  The 3 launches of
// an isolated 96^3 root's solve 51.3 -> 44.9 us, a 1 M Plummer step of three
// nested levels 808 -> 746, 32 grids of 128^3 742 -> 734, a two-level 64^3 step
// replayed as a graph 94.0 -> 91.4.  Letting the next kernel's CTAs in early
// (griddepcontrol.launch_dependents) costs more than it gives: the cosmological
// step 10.2 -> 11.6 ms, that graph 99.5 -> 123 us.
// The block index comes out of the same instruction sequence, so that every
// address a kernel forms from it, and with it every load, depends on the wait
// (loads through __restrict__ pointers may otherwise be moved across it).  The
// exceptions are the level and pointer tables of the all-level kernels (levels,
// gmfs, accs and the root's entry in them): no kernel writes those, and the
// copies that do come before the predecessor's own wait or after its end.
__device__ __forceinline__ unsigned begin_kernel() {
    unsigned block;
    asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, %%ctaid.x;" : "=r"(block) : : "memory");
    return block;
}
template <typename... KA, typename... A>
cudaError_t launch_kernel(void (*kernel)(KA...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t s,
                          A... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

// ---------------------------------------------------------------------------
// launchers (each returns the launch error)
// ---------------------------------------------------------------------------
// twiddles exp(-2 pi i t / L) for t < L, FP64 and FP32
cudaError_t launch_twiddles(double2* tw64, float2* tw32, int L, cudaStream_t s);

// Green's tables (FP64 octant), kind 0/1 directly, kind 2 from the real-space kernel
cudaError_t launch_green_table(int kind, const int M[3], double delta, double a_lev,
                               double a_par, int correction, int grad, double* out, double* scratch,
                               cudaStream_t s);
cudaError_t launch_to_f32(const double* in, float* out, long long n, cudaStream_t s);

// GMF: baryons (initialises every cell) then particles
cudaError_t launch_gas_init(const LevelDev& L, const GridDev* parent_grids,
                            const double* const* gas, const double* const* pgas,
                            int64_t* const* gmf, const Chunk* chunks, int n_chunks,
                            int F, cudaStream_t s);
cudaError_t launch_deposit(const LevelDev& L, const Particles& P, double half_dt, double box,
                           int F, int64_t* const* gmf, unsigned* status, cudaStream_t s);
// every level in one pass: levels[nl] and gmfs[nl] in device memory
cudaError_t launch_deposit_levels(const LevelDev* levels, int nl, double root_cells, bool overlap, const Particles& P,
                                  double half_dt, double box, int F, int64_t* const* const* gmfs, unsigned* status,
                                  cudaStream_t s);

// FFT passes of one level (T = float or double)
struct FftArgs {
    const GridDev* g;
    const Chunk* chunks;
    int n_chunks;
    const void* tw;        // complex twiddle arena of the precision
    const void* tab;       // table arena of the precision
    void* wsA;
    void* wsB;
    int F;
    size_t smem;
    int threads;           // threads per CTA: 128 or 256
    unsigned* status;      // device status word (bounded waits that ran out), or null
    int inject_wait = 0;   // fault injection: the x-forward bulk copy's wait runs out
    int comp = 0;          // spectral gradient: component of the z / xi passes (0 phi, 1-3 A_x..A_z)
};
cudaError_t fft_configure();

// Particle processing order (k_order.cu): a counting sort of the particle
// indices by root-level bin (cubes of 2^shift root cells, nb bins per axis) of
// their drifted positions into perm; count holds nb^3 bins, sums
// order_scan_chunks(nb^3) <= 1024 entries, key and rank n entries each.
int order_scan_chunks(int nbins);
cudaError_t launch_order(const LevelDev& root, const Particles& P, double half_dt, int shift, int nb,
                         unsigned* count, unsigned* sums, unsigned* key, unsigned* rank, int* perm, cudaStream_t s);
template <typename T>
cudaError_t launch_fft_xf(const FftArgs& a, const int64_t* const* gmf, cudaStream_t s);
template <typename T>
cudaError_t launch_fft_yf(const FftArgs& a, cudaStream_t s);
template <typename T>
cudaError_t launch_fft_z(const FftArgs& a, cudaStream_t s);
template <typename T>
cudaError_t launch_fft_yi(const FftArgs& a, cudaStream_t s);
// the z pass of a spectral-gradient component (a.comp in 1..3): the table
// times -i D_comp between the forward and the inverse transform
template <typename T>
cudaError_t launch_fft_zgrad(const FftArgs& a, cudaStream_t s);
template <typename T>
cudaError_t launch_fft_xi(const FftArgs& a, void* const* phis, cudaStream_t s);
// The passes with a compile-time plan of length L (fast_length), by kernel:
// the y forward, z (with the table) and y inverse column passes, the x forward
// and x inverse, the z pass of spectral component a.comp, and (FP32) the fused
// plane kernels: x + y forward over one z plane (k_xy_fast) of a grid with
// M0 = M1 = L, and y + x inverse over one window plane (k_yx_fast) for grids
// whose window fits the transform (W1 <= M1).
enum { kFastYf = 0, kFastZ, kFastYi, kFastXf, kFastXi, kFastZg, kFastXy, kFastYx, kFastKernels };
// threads of a plane kernel: 384, and 512 for the x + y forward where two planes
// fit an SM (32 grids of L = 150: 368 -> 353 us; the inverse loses, 218 -> 244, as
// does an isolated root of L = 192 with one plane per SM)
constexpr int kFastXyThreads = 384;
// the plane (L rows x L/2 + 1 columns) and the twiddles
constexpr size_t fast_xy_smem(int L) { return (size_t)(L * (L / 2 + 1) + L) * sizeof(float2); }
constexpr int fast_xy_threads(int kernel, int L) {
    return kernel == kFastXy && 2 * (fast_xy_smem(L) + 1024) <= (size_t)227 * 1024 ? 512 : kFastXyThreads;
}
inline bool fast_xy_length(int L) { return fast_length(L, false) && fast_xy_smem(L) <= (size_t)kFftSmemLimit; }
// plan 0 runs the fused planes for M0 = M1 = L from 70 to 192 (plan 2: wherever
// a plane fits).  Measured, unfused against fused, one level's five passes in
// us: 8 grids of L = 84 65.8 / 51.2, 27 of them 166.5 / 165.1, 8 of 120 148.9 /
// 133.5, 1 of 150 63.7 / 43.1, 27 of 150 1028 / 765, 8 of 160 451 / 319, 8 of
// 192 766 / 678, an isolated 96^3 root (192) 71.8 / 53.4.  Above 192 one plane
// fills an SM and the passes one by one are faster (8 of 216: 950 / 1047, a
// periodic 200^3 root 127 / 157).  Below 70 plan 0 keeps its separate passes,
// as it always had, although the planes are faster there too (1 of 45: 26.6 /
// 16.5): plan 2 asks for them.
inline bool fast_xy_default(int L) { return L >= 70 && L <= 192; }
cudaError_t launch_fft_fast(int kernel, bool f64, int L, const FftArgs& a, const int64_t* const* gmf,
                            void* const* phis, cudaStream_t s);
// allows the kernel its shared memory (once per kernel and device before its
// first launch; not inside a stream capture)
cudaError_t configure_fft_fast(int kernel, bool f64, int L);

// accelerations + parent carry for the four-point and spectral gradients (the
// two-point one runs launch_accel): the four-point one on flat ranges of blocks,
// the spectral one on launch_accel's columns
template <typename T>
cudaError_t launch_accel_var(const LevelDev& L, const GridDev* parent_grids, const void* const* phis,
                               const void* const* pphi, const void* const* pacc, void* const* phi,
                               void* const* acc, const Chunk* chunks, int n_chunks, int grad, int zs,
                               cudaStream_t s);

// FD accelerations + parent carry (two-point; a chunk is kAccThreads columns of
// blocks of one segment of zs blocks along z); TSC interpolation
template <typename T>
cudaError_t launch_accel(const LevelDev& L, const GridDev* parent_grids, const void* const* phis,
                         const void* const* pphi, const void* const* pacc, void* const* phi,
                         void* const* acc, const Chunk* chunks, int n_chunks, int zs,
                         cudaStream_t s);
template <typename T>
cudaError_t launch_interp(const LevelDev& L, const LevelDev* finer, const Particles& P,
                          double half_dt, const void* const* acc, void* out, cudaStream_t s);
// every level in one pass: levels[nl] and accs[nl] in device memory
template <typename T>
cudaError_t launch_interp_levels(const LevelDev* levels, int nl, const Particles& P, double half_dt,
                                 const void* const* const* accs, void* out, cudaStream_t s);

// one leapfrog step of the particles (k_evolve.cu); acc: 3n values of T
template <typename T>
cudaError_t launch_kick_drift(long long n, double* x, double* y, double* z, double* vx, double* vy, double* vz,
                              const void* acc, double dt, cudaStream_t s);

}  // namespace apm
