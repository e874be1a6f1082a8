// k_deposit.cu -- gravitating-mass field (GMF) of every grid of a level (Sec. 2):
// baryons (interior gas, parent gas copied onto the border) initialise every
// cell, then each particle, drifted half a timestep, adds its 27 TSC charges
// in 64-bit fixed point with integer atomics.  Integer addition is exact and
// associative, so the field is bit-identical for any particle order and any
// atomic interleaving.  Every floating-point step uses explicitly rounded
// intrinsics (no contraction), so the charges equal a plain IEEE evaluation.
#include "apm_internal.cuh"

namespace apm {
namespace {


// no baryons: the CTA's rows are one flat range of n zeros, written as
// 16-byte stores when the range starts 16-byte aligned
__device__ __noinline__ void zero_range(int64_t* __restrict__ z, long long n) {
    long long i0 = 0;
    if ((reinterpret_cast<size_t>(z) & 15) == 0) {
        longlong2* __restrict__ z2 = reinterpret_cast<longlong2*>(z);
        for (long long i = threadIdx.x; i < n / 2; i += blockDim.x) z2[i] = make_longlong2(0, 0);
        i0 = n & ~1LL;
    }
    for (long long i = i0 + threadIdx.x; i < n; i += blockDim.x) z[i] = 0;
}

// One CTA per batch of `rows` GMF rows (a row: G0 cells along x at fixed y, z).
__global__ void __launch_bounds__(256) k_gas_init(LevelDev L, const GridDev* __restrict__ pgrids,
                           const double* const* __restrict__ gas,
                           const double* const* __restrict__ pgas, int64_t* const* __restrict__ gmf,
                           const Chunk* __restrict__ chunks, int F) {
    const unsigned block = begin_kernel();
    const Chunk c = chunks[block];
    const GridDev& g = L.g[c.grid];
    const int G0 = g.G[0], G1 = g.G[1];
    const int nrows = G1 * g.G[2];
    const double* own = gas ? gas[c.grid] : nullptr;
    const double* par = (pgas && g.parent >= 0) ? pgas[g.parent] : nullptr;
    int64_t* __restrict__ out = gmf[c.grid];
    const int B = (G0 - g.N[0]) / 2;
    const int r0 = c.tile * g.rows_gas;
    const int r1 = min(nrows, r0 + g.rows_gas);
    const GridDev* p = par ? &pgrids[g.parent] : nullptr;
    if (!own && !par) {
        zero_range(out + (long long)r0 * G0, (long long)(r1 - r0) * G0);
        return;
    }
    const double scale = ldexp(1.0, F);
    const double vol = __dmul_rn(__dmul_rn(g.delta, g.delta), g.delta);
    // when delta is a power of two, 2^e, the two products are exact exponent
    // shifts and rint((rho delta^3) 2^F) = rint(rho 2^(F + 3e)): one FP64 addition,
    // or from 2^50 units up integer operations (scaled_rint), where the products and
    // the conversion would bound the pass (256^3 cells of half a unit mass: 226 us,
    // so 116; small ones 92).  The products remain for other cell sizes and beyond
    // 2^62.
    const unsigned long long db = (unsigned long long)__double_as_longlong(g.delta);
    const int de = (int)((db >> 52) & 0x7FF);
    const bool pow2 = (db & 0xFFFFFFFFFFFFFULL) == 0 && de > 0 && de < 0x7FF;
    const int K = F + 3 * (de - 1023);
    int last = -1, cy = 0, cz = 0;
    bool yz_in = false;
    for (RowWalk it(r0, G0); it.r < r1; it.next()) {
        const int r = it.r, x = it.x;
        int64_t* row = out + (long long)r * G0;
        if (r != last) {
            last = r;
            cy = r % G1 - B;
            cz = r / G1 - B;
            yz_in = cy >= 0 && cy < g.N[1] && cz >= 0 && cz < g.N[2];
        }
        const int cx = x - B;
        double rho = 0.0;
        if (yz_in && cx >= 0 && cx < g.N[0]) {
            if (own) rho = own[cx + (long long)g.N[0] * (cy + (long long)g.N[1] * cz)];
        } else if (par) {
            // parent cell floor(c / 2): the refinement factor is 2 (checked on the host);
            // past an isolated root's faces (the only border cells with no parent
            // cell, checked on the host) there are no baryons
            long long px = ((g.start[0] + cx) >> 1) - p->start[0];
            long long py = ((g.start[1] + cy) >> 1) - p->start[1];
            long long pz = ((g.start[2] + cz) >> 1) - p->start[2];
            if (px >= 0 && px < p->N[0] && py >= 0 && py < p->N[1] && pz >= 0 && pz < p->N[2])
                rho = par[px + (long long)p->N[0] * (py + (long long)p->N[1] * pz)];
        }
        if (APM_IN_BOUNDS((long long)r * G0 + x, g.cells_gmf, L.status)) {
            bool ok = false;
            long long v = pow2 ? scaled_rint(rho, K, ok) : 0;
            if (!ok) v = __double2ll_rn(__dmul_rn(__dmul_rn(rho, vol), scale));
            row[x] = v;
        }
    }
}


// GMF-local index of one cloud cell per axis under the grid's edge rule
// (mode 0 drop: -1 when outside, 1 fold, 2 wrap)
// (on the periodic root the centre cell is in [0, G), so v is in [-1, G])
template <typename I>
__device__ __forceinline__ int edge_rule(I v, int G, int mode) {
    if (mode == 1) return v < 0 ? 0 : (v >= G ? G - 1 : (int)v);
    if (mode == 2) return (int)(v < 0 ? v + G : (v >= G ? v - G : v));
    return (v < 0 || v >= G) ? -1 : (int)v;
}

// CTA size and minimum resident CTAs per SM of the particle deposit
#ifndef APM_DEP_THREADS
#define APM_DEP_THREADS 128
#endif
#ifndef APM_DEP_MIN_CTAS
#define APM_DEP_MIN_CTAS 8
#endif
constexpr int kDepThreads = APM_DEP_THREADS;
static_assert(kDepThreads % 32 == 0, "the deposit works by whole warps");

// ---- the particles' deposit: a warp sends rows of clouds ----
// What bounds the deposit is the 64-bit reductions, in the SM's load/store unit
// and in L2, and both serve them by 32-byte sector: a warp instruction whose 32
// lanes add into one cell each of 32 particles' clouds touches 32 sectors, one
// whose lanes add 3 neighbouring cells of 8 particles 10 to 12 (5 for particles
// stored in x order, whose rows adjoin).  Probed with red.global.add.u64 on a
// 512^3 field, 16.8 M particles: 265 against 470 G reductions/s in lattice
// order, 59 against 88 G/s at random places.
// So each lane computes its own particle's charges into shared memory, 9 (one
// z layer of the cloud) at a time, and the warp then sends them 8 particles at a
// time, lane 8 a + p the cell a of particle p in each (y, z) row.  The kernel
// waits on latency: a layer at a time takes 4.6 KB of shared memory a warp and
// 64 registers a thread, 32 warps per SM (all 27 charges at once: 20 warps and
// 1.74 ms where this took 1.46).  Integer addition is exact and associative:
// the field does not depend on the arrangement.  Pitch 40: lanes on 32
// particles (stores) and on 3 x 8 (loads) fall into distinct banks.
// All levels, before (one particle per thread, x neighbours' columns merged in
// registers) -> now: 16.8 M lattice particles on 512^3 with two refined levels
// 1.82 -> 1.43 ms; 4.2 M random ones on 256^3 1.23 -> 0.78; a Plummer sphere of
// 1 M through three nested levels 0.96 -> 0.54.
constexpr int kChargePitch = 40;
struct WarpCharges {
    union {                            // charge of cell a + 3 b of the layer, of each lane's particle
        unsigned narrow[9][kChargePitch];
        unsigned long long wide[9][kChargePitch];
    };
    unsigned off[9][kChargePitch];     // cx[3], G0 cy[3], G0 G1 cz[3]; kNoCell: outside
    int64_t* base[32];                 // the mass field of each lane's grid
};
constexpr unsigned kNoCell = 0x80000000u;   // mass fields hold fewer than 2^31 cells

// This lane's particle's charges, layer by layer: ((|M| wx) wy) wz for the 26
// outer cells, every product rounded half up on the scale 2^63, the centre cell
// |M| minus the others, all with the sign of M; the middle layer, which holds the
// centre, comes last.  V = unsigned holds every charge of a mass in [2^9, 2^32)
// (narrow_mass): none exceeds it, as the weights sum to one, and the centre cell's
// is positive, as its weight is at least 1/8 (1/2 an axis) and the 26 others are
// rounded up by less than 2 units each.  The centre of a smaller mass may be
// negative (M = 1 on a cell corner: 7 charges of 1, centre -6).
constexpr long long kMinNarrow = 512;
__device__ __forceinline__ bool narrow_mass(long long M) {
    return (unsigned long long)(M - kMinNarrow) < (1ULL << 32) - (unsigned long long)kMinNarrow;
}
__device__ __forceinline__ unsigned mul63w(unsigned a, unsigned long long b) { return wmul63_32(a, b); }
__device__ __forceinline__ unsigned long long mul63w(unsigned long long a, unsigned long long b) {
    return wmul63(a, b);
}
template <typename V> struct LaneCharges {
    V mxy[9];        // (|M| wx) wy of cell a + 3 b
    V centre;        // |M| minus the outer charges so far (64 bits: modulo 2^64)
    bool negative;
    __device__ __forceinline__ void start(long long M, const unsigned long long w[3][3]) {
        negative = M < 0;
        centre = (V)(M < 0 ? -M : M);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const V mx = mul63w(centre, w[0][a]);
#pragma unroll
            for (int b = 0; b < 3; ++b) mxy[a + 3 * b] = mul63w(mx, w[1][b]);
        }
    }
    // put(k, charge) for the cells k = a + 3 b of layer c
    template <class PUT>
    __device__ __forceinline__ void layer(int c, const unsigned long long w[3][3], PUT put) {
        const unsigned long long wz = c == 0 ? w[2][0] : (c == 1 ? w[2][1] : w[2][2]);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if (k == 4 && c == 1) continue;
            V v = mul63w(mxy[k], wz);
            centre -= v;
            if (sizeof(V) == 8 && negative) v = (V)0 - v;
            put(k, v);
        }
        if (c == 1) put(4, sizeof(V) == 8 && negative ? (V)0 - centre : centre);
    }
};

// the cells of this lane's cloud in grid g (centre cell ic) as summable offsets
// (a centre cell beyond [-2, G + 1], an isolated root's particle outside the box,
// folds like these do)
__device__ __forceinline__ int local_centre(const GridDev& g, const long long ic[3], int j) {
    return (int)min(max(ic[j] - g.lo[j], -2LL), (long long)g.G[j] + 1);
}
__device__ __forceinline__ void lane_cells(WarpCharges& s, int lane, const GridDev& g, const long long ic[3],
                                           unsigned* __restrict__ status) {
    const unsigned st[3] = {1u, (unsigned)g.G[0], (unsigned)g.G[0] * (unsigned)g.G[1]};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int G = g.G[j], r = local_centre(g, ic, j);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int v = edge_rule(r + k - 1, G, g.mode);
            s.off[3 * j + k][lane] = v >= 0 && APM_IN_BOUNDS(v, G, status) ? st[j] * (unsigned)v : kNoCell;
        }
    }
}

// layer c of the clouds of the lanes in `live` (a warp mask, the same on every lane)
template <bool WIDE>
__device__ __forceinline__ void send_layer(const WarpCharges& s, int lane, unsigned live, int c) {
    const int a = lane >> 3, p = lane & 7;
    if (a == 3) return;
#pragma unroll 2
    for (int k0 = 0; k0 < 32; k0 += 8) {
        const int k = k0 + p;
        if (!((live >> k) & 1u)) continue;
        const unsigned ox = s.off[a][k], oz = s.off[6 + c][k], xz = ox + oz, out = ox | oz;
        int64_t* const base = s.base[k];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const unsigned o = s.off[3 + b][k];
            const unsigned long long q = WIDE ? s.wide[a + 3 * b][k] : s.narrow[a + 3 * b][k];
            // a particle on a cell face has charges of zero (19 of 27 on a corner): not
            // sent (16.8 M corner particles on 256^3: 1.01 -> 0.92 ms)
            if ((out | o) < kNoCell && q != 0)
                asm volatile("red.global.add.u64 [%0], %1;" ::"l"(base + (xz + o)), "l"(q));
        }
    }
}

// the warp's clouds in one grid each, layer by layer; X: this lane's position on
// a level with P fraction bits
template <typename V>
__device__ __forceinline__ void send_clouds(WarpCharges& s, int lane, bool act, long long M, long long x, long long y,
                                            long long z, int P) {
    constexpr bool kWide = sizeof(V) == 8;
    const unsigned live = __ballot_sync(0xffffffffu, act);
    unsigned long long w[3][3];
    tsc_fixed(x, P, w[0]);
    tsc_fixed(y, P, w[1]);
    tsc_fixed(z, P, w[2]);
    LaneCharges<V> q;
    q.start(M, w);
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const int c = k == 0 ? 0 : 3 - k;   // 0, 2, 1
        if (act)
            q.layer(c, w, [&](int j, V v) {
                if constexpr (kWide) s.wide[j][lane] = v;
                else s.narrow[j][lane] = v;
            });
        __syncwarp();
        send_layer<kWide>(s, lane, live, c);
        __syncwarp();
    }
}
// out of line: the registers of the 64-bit charges stay out of the usual path
__device__ __noinline__ void send_wide_clouds(WarpCharges& s, int lane, bool act, long long M, long long x, long long y,
                                              long long z, int P) {
    send_clouds<unsigned long long>(s, lane, act, M, x, y, z, P);
}

// This lane's cloud straight into the candidate grids [e0, e1) (list null: the
// root), one reduction per cell; UNROLL of the three layers
template <typename V, int UNROLL>
__device__ __forceinline__ void send_direct(const GridDev* __restrict__ grids, const int* __restrict__ list, int e0, int e1,
                                         long long M, long long x, long long y, long long z, int P,
                                         int64_t* const* __restrict__ gmf, unsigned* __restrict__ status) {
    const long long ic[3] = {x >> P, y >> P, z >> P};
    unsigned long long w[3][3];
    tsc_fixed(x, P, w[0]);
    tsc_fixed(y, P, w[1]);
    tsc_fixed(z, P, w[2]);
    for (int e = e0; e < e1; ++e) {
        const int gi = list ? list[e] : 0;
        const GridDev& g = grids[gi];
        const unsigned st[3] = {1u, (unsigned)g.G[0], (unsigned)g.G[0] * (unsigned)g.G[1]};
        unsigned off[3][3];
        bool touches = true;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int G = g.G[j], r = local_centre(g, ic, j);
            touches = touches && (g.mode != 0 || (r >= -1 && r <= G));
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int v = edge_rule(r + k - 1, G, g.mode);
                off[j][k] = v >= 0 && APM_IN_BOUNDS(v, G, status) ? st[j] * (unsigned)v : kNoCell;
            }
        }
        if (!touches) continue;   // listed by its tile only
        int64_t* __restrict__ const out = gmf[gi];
        LaneCharges<V> q;
        q.start(M, w);
#pragma unroll UNROLL
        for (int k = 0; k < 3; ++k) {
            const int c = k == 0 ? 0 : 3 - k;   // 0, 2, 1
            const unsigned oz = c == 0 ? off[2][0] : (c == 1 ? off[2][1] : off[2][2]);
            q.layer(c, w, [&](int j, V v) {
                const unsigned ox = off[0][j % 3], oy = off[1][j / 3];
                if ((ox | oy | oz) < kNoCell && v != 0)
                    asm volatile("red.global.add.u64 [%0], %1;" ::"l"(out + (ox + oy + oz)), "l"((unsigned long long)v));
            });
        }
    }
}

__device__ __forceinline__ bool candidates(const LevelDev& L, const long long ic[3], int& e0, int& e1);
// the cloud of a lane with more candidates on level L into those after the first
__device__ __forceinline__ void deposit_rest(const LevelDev& L, const long long X[3], long long M,
                                             int64_t* const* __restrict__ gmf, unsigned* __restrict__ status) {
    const int P = L.frac_bits;
    const long long ic[3] = {X[0] >> P, X[1] >> P, X[2] >> P};
    int e0, e1;
    candidates(L, ic, e0, e1);
    // (64-bit charges for every mass: the narrow ones round the same way)
    send_direct<unsigned long long, 1>(L.g, L.map.dep_list, e0 + 1, e1, M, X[0], X[1], X[2], P, gmf, status);
}

// How a launch sends its clouds: in rows; in rows, and straight into the candidate
// grids after the first, on levels with overlapping borders (rows for them would be
// mostly empty: 200000 random particles over 8 touching grids 72 -> 70 us, with
// 64-bit charges 92 -> 86); in bin order, like that where no box gathers them; all
// straight, which is the shorter way where a launch leaves most schedulers a warp or
// none.  A loop over the candidates in the rows' kernel spills registers there (1 M
// random particles on 256^3 246 us with it, 227 without; a lattice on 192^3 103, 98).
enum DepositWay { kRows, kRowsOverlap, kOrdered, kDirect };

// the candidate grids [e0, e1) of level L's tile lists for the centre cell ic
// (the root: [0, 1)); false when there is none
__device__ __forceinline__ bool candidates(const LevelDev& L, const long long ic[3], int& e0, int& e1) {
    e0 = 0;
    e1 = 1;
    if (L.is_root) return true;
    const TileMap& m = L.map;
    long long t[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const long long rel = ic[j] - m.lo[j];
        if (rel < 0) return false;
        t[j] = rel >> m.shift;
        if (t[j] >= m.nt[j]) return false;
    }
    const long long tile = t[0] + (long long)m.nt[0] * (t[1] + (long long)m.nt[1] * t[2]);
    e0 = m.dep_off[tile];
    e1 = m.dep_off[tile + 1];
    return e0 != e1;
}

// ---- particles in bin order: a CTA's clouds gathered in a box ----
// In bin order a CTA's particles lie close together, and where many share cells
// (a halo's core) it adds their charges in shared memory and sends one reduction
// per cell of the box around them, where the box of its clouds in one grid holds at
// most kBoxPerParticle cells for each of its particles (and fits the row charges'
// memory); elsewhere the warps send their rows.  A sum is two 32-bit words: of
// 32-bit charges the low and the high halves (at most 128 particles add less than
// 2^23 to either, and no carry is waited for), of 64-bit ones the low word, whose
// carry goes to the high one.  Integer sums do not depend on the order: the same
// field.  Rows only -> boxes, 1 M particles: a Plummer sphere on 256^3 281 -> 132
// us, on 64^3 570 -> 114, on 64^3 with one nested level 864 -> 188, through three
// levels 562 -> 344; at random places on 256^3 180 -> 181, on 64^3 139 -> 111.  With 6
// cells for each particle the two nested ones take 531 and 482, with 18 the same.
constexpr int kBoxCells = (int)(sizeof(WarpCharges) * (kDepThreads / 32) / 8);
#ifndef APM_DEP_BOX
#define APM_DEP_BOX 12
#endif
constexpr int kBoxPerParticle = APM_DEP_BOX;
struct Box {
    int lo[3], n[3];   // first cell (GMF-local, before the edge rule) and extents
    int cells;         // 0: none
    int gi;            // the grid
};
struct BoxShared {
    int lo[kDepThreads / 32][4], hi[kDepThreads / 32][4], count[kDepThreads / 32];
};
// the box of the CTA's acting lanes at the centre cells r of grid gi (lanes with
// other candidates beside it: one = false).  Every thread calls it.
__device__ __forceinline__ Box cta_box(BoxShared& b, bool act, bool one, int gi, const int r[3]) {
    constexpr unsigned kFull = 0xffffffffu;
    const int warp = threadIdx.x >> 5;
    const int v[4] = {r[0], r[1], r[2], one ? gi : -1};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int lo = __reduce_min_sync(kFull, act ? v[j] : 0x7fffffff);
        const int hi = __reduce_max_sync(kFull, act ? v[j] : -0x7fffffff);
        if ((threadIdx.x & 31) == 0) {
            b.lo[warp][j] = lo;
            b.hi[warp][j] = hi;
        }
    }
    const int count = __popc(__ballot_sync(kFull, act));
    if ((threadIdx.x & 31) == 0) b.count[warp] = count;
    __syncthreads();
    int lo[4], hi[4], total = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        lo[j] = 0x7fffffff;
        hi[j] = -0x7fffffff;
#pragma unroll
        for (int w = 0; w < kDepThreads / 32; ++w) {
            lo[j] = min(lo[j], b.lo[w][j]);
            hi[j] = max(hi[j], b.hi[w][j]);
        }
    }
#pragma unroll
    for (int w = 0; w < kDepThreads / 32; ++w) total += b.count[w];
    __syncthreads();   // read by every warp
    Box x;
    x.gi = lo[3];
    x.cells = 0;
    if (total == 0 || lo[3] < 0 || lo[3] != hi[3]) return x;
    long long cells = 1;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        x.lo[j] = lo[j] - 1;
        x.n[j] = hi[j] - lo[j] + 3;
        cells *= x.n[j];   // extents below 2^21
    }
    if (cells <= min(kBoxCells, kBoxPerParticle * total)) x.cells = (int)cells;
    return x;
}
// this lane's cloud (centre cell r) into the box
template <typename V>
__device__ __forceinline__ void box_add(unsigned* __restrict__ lo, unsigned* __restrict__ hi, const Box& x,
                                        const int r[3], long long M, const unsigned long long w[3][3]) {
    LaneCharges<V> q;
    q.start(M, w);
    const int n01 = x.n[0] * x.n[1];
    const int first = (r[0] - 1 - x.lo[0]) + x.n[0] * (r[1] - 1 - x.lo[1]) + n01 * (r[2] - 1 - x.lo[2]);
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const int c = k == 0 ? 0 : 3 - k;   // 0, 2, 1
        q.layer(c, w, [&](int j, V v) {
            const int at = first + c * n01 + (j % 3) + x.n[0] * (j / 3);
            if constexpr (sizeof(V) == 4) {
                if (v & 0xffffu) atomicAdd(lo + at, v & 0xffffu);
                if (v >> 16) atomicAdd(hi + at, v >> 16);
            } else {
                const unsigned l = (unsigned)v;
                const unsigned old = atomicAdd(lo + at, l);
                const unsigned h = (unsigned)(v >> 32) + (old + l < old ? 1u : 0u);
                if (h) atomicAdd(hi + at, h);
            }
        });
    }
}
// every acting lane's cloud into the box, then one reduction per cell that is not
// zero; words: kBoxCells low and high words.  Every thread calls it.
__device__ __forceinline__ void box_deposit(unsigned* __restrict__ words, const Box& x, const GridDev& g, bool act,
                                            const int r[3], long long M, const long long X[3], int P,
                                            int64_t* __restrict__ out, unsigned* __restrict__ status) {
    unsigned* const lo = words;
    unsigned* const hi = words + x.cells;
    for (int k = threadIdx.x; k < 2 * x.cells; k += kDepThreads) words[k] = 0u;
    // one width of charges for the CTA
    const bool wide = __syncthreads_or(act && M != 0 && !narrow_mass(M));
    if (act && M != 0) {
        unsigned long long w[3][3];
#pragma unroll
        for (int j = 0; j < 3; ++j) tsc_fixed(X[j], P, w[j]);
        if (wide) box_add<unsigned long long>(lo, hi, x, r, M, w);
        else box_add<unsigned>(lo, hi, x, r, M, w);
    }
    __syncthreads();
    const unsigned G0 = g.G[0], G01 = (unsigned)g.G[0] * (unsigned)g.G[1];
    for (int k = threadIdx.x; k < x.cells; k += kDepThreads) {
        const unsigned long long v =
            wide ? ((unsigned long long)hi[k] << 32 | lo[k]) : ((unsigned long long)hi[k] << 16) + lo[k];
        if (v == 0) continue;
        const int yz = k / x.n[0], cz = yz / x.n[1];
        const int c0 = edge_rule(x.lo[0] + k - yz * x.n[0], g.G[0], g.mode);
        const int c1 = edge_rule(x.lo[1] + yz - cz * x.n[1], g.G[1], g.mode);
        const int c2 = edge_rule(x.lo[2] + cz, g.G[2], g.mode);
        if ((c0 | c1 | c2) < 0) continue;
        const unsigned at = (unsigned)c0 + G0 * (unsigned)c1 + G01 * (unsigned)c2;
        if (APM_IN_BOUNDS(at, g.cells_gmf, status))
            asm volatile("red.global.add.u64 [%0], %1;" ::"l"(out + at), "l"(v));
    }
    __syncthreads();   // the words are the warps' row charges too
}

// The deposit into the grids of one level: this lane's particle at fixed-point
// position X with integer mass M (ok false: none).  Every lane of the warp calls
// it, kOrdered every thread of the CTA.  False when this lane's particle is not a candidate of
// the level (then it is none of a finer level's either: finer GMF boxes lie
// inside the interiors of their parents).
template <DepositWay WAY>
__device__ __forceinline__ bool deposit_level_warp(WarpCharges* charges, BoxShared* box, const LevelDev& L,
                                                   const long long X[3], long long M, bool ok, bool outside, bool& more,
                                                   int64_t* const* __restrict__ gmf,
                                                   unsigned* __restrict__ status) {
    more = false;
    constexpr unsigned kFull = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int PB = L.frac_bits;
    long long ic[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) ic[j] = X[j] >> PB;
    int e0 = 0, e1 = 0;
    ok = ok && candidates(L, ic, e0, e1);
    if constexpr (WAY == kOrdered) {
        if (!__syncthreads_or(ok)) return false;
        const int gi = !ok ? 0 : (L.is_root ? 0 : L.map.dep_list[e0]);
        const GridDev& g = L.g[gi];
        const int r[3] = {local_centre(g, ic, 0), local_centre(g, ic, 1), local_centre(g, ic, 2)};
        const Box x = cta_box(*box, ok, e1 - e0 == 1, gi, r);
        if (x.cells > 0) {
            if (ok && g.mode == 1 && outside) atomicOr(status, kStOutOfBox);
            box_deposit(reinterpret_cast<unsigned*>(charges), x, L.g[x.gi], ok, r, M, X, PB, gmf[x.gi], status);
            return ok;
        }
    }
    if (!__any_sync(kFull, ok)) return false;
    // one charge width for the whole warp (the 32-bit products round the same way)
    const bool wide = __any_sync(kFull, ok && M != 0 && !narrow_mass(M));
    if (!ok) e1 = e0;
    if (ok && outside) atomicOr(status, kStOutOfBox);
    const int* const list = L.is_root ? nullptr : L.map.dep_list;
    if constexpr (WAY == kDirect) {
        if (e0 < e1 && M != 0) {
            if (wide) send_direct<unsigned long long, 3>(L.g, list, e0, e1, M, X[0], X[1], X[2], PB, gmf, status);
            else send_direct<unsigned, 3>(L.g, list, e0, e1, M, X[0], X[1], X[2], PB, gmf, status);
        }
        return ok;
    }
    WarpCharges& s = charges[threadIdx.x >> 5];
    const bool act = e0 < e1;
    if (act) {
        const int gi = list ? list[e0] : 0;
        lane_cells(s, lane, L.g[gi], ic, status);
        s.base[lane] = gmf[gi];
    }
    // a particle without mass sends nothing
    if (wide) send_wide_clouds(s, lane, act && M != 0, M, X[0], X[1], X[2], PB);
    else send_clouds<unsigned>(s, lane, act && M != 0, M, X[0], X[1], X[2], PB);
    more = e0 + 1 < e1 && M != 0;
    return ok;
}

// drifted coordinates, fixed-point position and integer mass of particle p;
// false (and the overflow flag) when |m 2^F| >= 2^62
__device__ __forceinline__ bool particle_fixed(const LevelDev& L, const Particles& P, long long p,
                                               double half_dt, double box, int F, long long X[3],
                                               long long* M, bool* outside, unsigned* __restrict__ status) {
    const double xd[3] = {drift_raw(P.x[p], P.vx[p], half_dt), drift_raw(P.y[p], P.vy[p], half_dt),
                          drift_raw(P.z[p], P.vz[p], half_dt)};
#pragma unroll
    for (int j = 0; j < 3; ++j) X[j] = fixed_position(xd[j], L);   // the same for every level
    bool ok;
    *M = scaled_rint(P.m[p], F, ok);   // rint(m 2^F)
    if (!ok) {
        atomicOr(status, kStOverflow);
        return false;
    }
    // isolated root only: a drifted particle outside [0, box) is flagged (its cloud folds)
    *outside = L.g[0].mode == 1 && L.is_root &&
               !(xd[0] >= 0.0 && xd[0] < box && xd[1] >= 0.0 && xd[1] < box && xd[2] >= 0.0 && xd[2] < box);
    return true;
}

// slot i's particle for the deposit into one level: its fixed-point position
// and integer mass; false when it is none of the level's (the candidate test
// first on refined levels: most particles leave there) or its mass overflows
__device__ __forceinline__ bool particle_of_level(const LevelDev& L, const Particles& P, long long i, double half_dt,
                                                  double box, int F, long long X[3], long long* M, bool* outside,
                                                  unsigned* __restrict__ status) {
    const long long p = P.at(i);
    *outside = false;
    if (L.is_root) return particle_fixed(L, P, p, half_dt, box, F, X, M, outside, status);
    const double xd[3] = {drift_raw(P.x[p], P.vx[p], half_dt), drift_raw(P.y[p], P.vy[p], half_dt),
                          drift_raw(P.z[p], P.vz[p], half_dt)};
#pragma unroll
    for (int j = 0; j < 3; ++j) X[j] = fixed_position(xd[j], L);
    const long long ic[3] = {X[0] >> L.frac_bits, X[1] >> L.frac_bits, X[2] >> L.frac_bits};
    int e0, e1;
    if (!candidates(L, ic, e0, e1)) return false;
    bool ok;
    *M = scaled_rint(P.m[p], F, ok);
    if (!ok) atomicOr(status, kStOverflow);
    return ok;
}

// this thread's slot: in the caller's order CTA after CTA; in bin order spread over
// the bins (deposit_stride, coprime to the number of CTAs).  spread: the warp's 32
// slots transposed, lane 8 j + p taking slot 4 p + j, so that the 8 clouds an
// instruction sends are every fourth one
__device__ __forceinline__ long long thread_slot(const Particles& P, unsigned b) {
    if (P.stride) b = (unsigned)((unsigned long long)b * P.stride % gridDim.x);
    unsigned t = threadIdx.x;
    if (P.spread) t = (t & ~31u) | (t & 7u) << 2 | (t >> 3 & 3u);
    return (long long)b * kDepThreads + t;
}

constexpr int dep_min_ctas(DepositWay way) { return way == kDirect ? 4 : APM_DEP_MIN_CTAS; }
// One level.
template <DepositWay WAY>
__global__ void __launch_bounds__(kDepThreads, dep_min_ctas(WAY)) k_deposit(LevelDev L, Particles P, double half_dt,
                                                 double box, int F,
                                                 int64_t* const* __restrict__ gmf,
                                                 unsigned* __restrict__ status) {
    const unsigned block = begin_kernel();
    __shared__ WarpCharges charges[kDepThreads / 32];
    __shared__ BoxShared cta[1];
    const long long i = thread_slot(P, block);
    long long X[3] = {0, 0, 0}, M = 0;
    bool outside = false;
    const bool ok = i < P.n && particle_of_level(L, P, i, half_dt, box, F, X, &M, &outside, status);
    bool more;
    deposit_level_warp<WAY>(charges, cta, L, X, M, ok, outside, more, gmf, status);
    if ((WAY == kRowsOverlap || WAY == kOrdered) && more) deposit_rest(L, X, M, gmf, status);
}

// Every level in one pass over the particles: the position and mass are
// converted once, then deposited level by level from the root down while the
// particle is a candidate.  levels: the LevelDev of each level; gmfs[l]: the
// GMF pointer table of level l.
template <DepositWay WAY>
__global__ void __launch_bounds__(kDepThreads, dep_min_ctas(WAY)) k_deposit_levels(
    const LevelDev* __restrict__ levels, int nl, Particles P, double half_dt, double box, int F,
    int64_t* const* const* __restrict__ gmfs, unsigned* __restrict__ status) {
    const unsigned block = begin_kernel();
    __shared__ WarpCharges charges[kDepThreads / 32];
    __shared__ BoxShared cta[1];
    const long long i = thread_slot(P, block);
    long long X[3] = {0, 0, 0}, M = 0;
    bool outside = false, ok = false;
    if (i < P.n) ok = particle_fixed(levels[0], P, P.at(i), half_dt, box, F, X, &M, &outside, status);
    unsigned rest = 0;   // levels (at most 21) with more candidates for this lane
    for (int l = 0; l < nl; ++l) {
        bool more;
        ok = deposit_level_warp<WAY>(charges, cta, levels[l], X, M, ok, l == 0 && outside, more, gmfs[l], status);
        if (more) rest |= 1u << l;
        if constexpr (WAY == kOrdered) {   // the CTA's box needs all its warps
            if (!__syncthreads_or(ok)) break;
        } else {
            if (!__any_sync(0xffffffffu, ok)) break;
        }
    }
    // after the levels, so that no call stands in their loop
    if constexpr (WAY == kRowsOverlap || WAY == kOrdered) {
        for (; rest; rest &= rest - 1) {
            const int l = __ffs(rest) - 1;
            deposit_rest(levels[l], X, M, gmfs[l], status);
        }
    }
}

}  // namespace

cudaError_t launch_gas_init(const LevelDev& L, const GridDev* parent_grids,
                            const double* const* gas, const double* const* pgas,
                            int64_t* const* gmf, const Chunk* chunks, int n_chunks,
                            int F, cudaStream_t s) {
    if (n_chunks <= 0) return cudaSuccess;
    return launch_kernel(k_gas_init, n_chunks, 256, 0, s, L, parent_grids, gas, pgas, gmf, chunks, F);
}

// In bin order the CTAs that run together would add into the same few cells
// where many particles share them and no box gathers them; a golden-ratio stride
// through the CTAs spreads them over the bins, and each CTA keeps its own bin's
// locality.  A Plummer sphere of 1 M through three nested levels 413 -> 344 us
// (caller's order 544); random places on 256^3 166 -> 182 (227).
// In the caller's order, where there are two particles or more to a root cell,
// neighbouring ones stored in spatial order share cells, and an instruction's
// reductions into one cell wait for one another: it sends every fourth particle
// instead.  A lattice of 8 to a cell on 128^3 1252 -> 1019 us, of 64 to a cell on
// 64^3 2248 -> 1437, of 4 to a cell on 128^3 608 -> 545 (947, 1366 and 504 now); of
// one to a cell on 256^3 1031 either way, and below that the neighbours' shared
// sectors are worth more (one to 8 cells there 168 -> 194).  In no spatial order it
// makes no difference.
static Particles deposit_order(Particles P, unsigned blocks, double cells) {
    P.stride = 0;
    P.spread = !P.perm && (double)P.n >= 2.0 * cells;
    if (P.perm && blocks > 2) {
        auto gcd = [](unsigned a, unsigned b) {
            while (b) {
                const unsigned t = a % b;
                a = b;
                b = t;
            }
            return a;
        };
        P.stride = (unsigned)(0.6180339887 * blocks) | 1u;
        while (gcd(P.stride, blocks) != 1) P.stride += 2;
    }
    return P;
}

// Straight up to 16384 particles (64-bit charges on an isolated 32^3 root 12.4 us in
// rows, 10.4 so; 20000 on a 60^3 root 12.4 in rows and 14.0 so), four times as many
// where levels overlap (8586 over 8 touching grids 33 us in rows and 23 so, 60000 39
// and 37, with 64-bit charges 41 and 25, 46 and 39).
constexpr long long kDirectParticles = 16384;
static DepositWay deposit_way(const Particles& P, bool overlap) {
    if (P.perm) return kOrdered;
    if (P.n <= (overlap ? 4 * kDirectParticles : kDirectParticles)) return kDirect;
    return overlap ? kRowsOverlap : kRows;
}

cudaError_t launch_deposit(const LevelDev& L, const Particles& P, double half_dt, double box,
                           int F, int64_t* const* gmf, unsigned* status, cudaStream_t s) {
    if (P.n <= 0) return cudaSuccess;
    unsigned blocks = (unsigned)((P.n + kDepThreads - 1) / kDepThreads);
    void (*const kernels[])(LevelDev, Particles, double, double, int, int64_t* const*, unsigned*) = {
        k_deposit<kRows>, k_deposit<kRowsOverlap>, k_deposit<kOrdered>, k_deposit<kDirect>};
    return launch_kernel(kernels[deposit_way(P, L.overlap != 0)], blocks, kDepThreads, 0, s, L,
                         deposit_order(P, blocks, L.root_cells), half_dt, box, F, gmf, status);
}

cudaError_t launch_deposit_levels(const LevelDev* levels, int nl, double root_cells, bool overlap, const Particles& P,
                                  double half_dt, double box, int F, int64_t* const* const* gmfs, unsigned* status,
                                  cudaStream_t s) {
    if (P.n <= 0 || nl <= 0) return cudaSuccess;
    unsigned blocks = (unsigned)((P.n + kDepThreads - 1) / kDepThreads);
    void (*const kernels[])(const LevelDev*, int, Particles, double, double, int, int64_t* const* const*, unsigned*) = {
        k_deposit_levels<kRows>, k_deposit_levels<kRowsOverlap>, k_deposit_levels<kOrdered>, k_deposit_levels<kDirect>};
    return launch_kernel(kernels[deposit_way(P, overlap)], blocks, kDepThreads, 0, s, levels, nl,
                         deposit_order(P, blocks, root_cells), half_dt, box, F, gmfs, status);
}

}  // namespace apm
