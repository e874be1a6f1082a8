// k_field.cu -- cell accelerations with the parent carry, and TSC interpolation
// of the accelerations back to the particles (Sec. 2.2, Sec. 2).
#include "apm_internal.cuh"

namespace apm {
namespace {

// acc_j(c) = -(phis(c+e_j) - phis(c-e_j)) / (2 delta) + I(parent acc_j)(c)
// phi(c)   = phis(c) + I(parent phi)(c),    c in [-1, N]^3
// I is the trilinear interpolation from the parent cell centres (Sec. 2.2), for
// R = 2: level cells 2k+1 and 2k+2 lie 1/4 and 3/4 of a parent cell above the
// centre of parent cell k, so they weigh parent cells (k, k+1) with (3/4, 1/4)
// and (1/4, 3/4).  The work unit is a 2x2x2 block of such cells: the 8 parent
// values of a field serve all 8 cells, interpolated separably (x, then y, then
// z).  Everything is evaluated in T; the weights are exact.
// A block may straddle the edge of [-1, N]: its outside cells are not written
// and the loads they would need are clamped into the window.
template <typename T>
__device__ __forceinline__ void lerp_block(const T q[2][2][2], T out[2][2][2]) {
    const T a = (T)0.75, b = (T)0.25;
    T x[2][2][2], y[2][2][2];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            x[dz][dy][0] = a * q[dz][dy][0] + b * q[dz][dy][1];
            x[dz][dy][1] = b * q[dz][dy][0] + a * q[dz][dy][1];
        }
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int cx = 0; cx < 2; ++cx) {
            y[dz][0][cx] = a * x[dz][0][cx] + b * x[dz][1][cx];
            y[dz][1][cx] = b * x[dz][0][cx] + a * x[dz][1][cx];
        }
#pragma unroll
    for (int cy = 0; cy < 2; ++cy)
#pragma unroll
        for (int cx = 0; cx < 2; ++cx) {
            out[0][cy][cx] = a * y[0][cy][cx] + b * y[1][cy][cx];
            out[1][cy][cx] = b * y[0][cy][cx] + a * y[1][cy][cx];
        }
}

__device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk2(double a, double b) { return make_double2(a, b); }

template <typename T>
__device__ __forceinline__ void load_parent(const T* __restrict__ f, unsigned base, int P0, unsigned P01,
                                            T q[2][2][2]) {
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) q[dz][dy][dx] = f[base + dx + dy * P0 + dz * P01];
}

// minimum resident CTAs per SM of the FP32 acceleration kernels: the two-point
// march wants its 128 registers (32 grids of 128^3: 324 us at 4 CTAs, 402 at 5,
// 490 at 6, 376 at 3), the others one block per thread
#ifndef APM_ACC_MIN_CTAS
#define APM_ACC_MIN_CTAS 4
#endif
template <typename T> struct AccMinCtas { static constexpr int march = APM_ACC_MIN_CTAS, value = 6; };
template <> struct AccMinCtas<double> { static constexpr int march = 1, value = 1; };

// The two-point difference.  What bounds it is the latency of its loads (and
// HBM: 0.60 of the measured copy rate with one block per thread).  A thread
// marches up z through zs blocks of one (x, y) column, so a block takes from the
// one below it the parent plane between them, interpolated in x and y, and the
// potential planes: 16 parent values and 16 loads of the potential a block
// instead of 32 and 24.  The next block's first plane is loaded with the current
// one (its centres are this block's upper z neighbours).
// 32 refined grids of 128^3: 391 -> 324 us (1566 MB: 4.0 -> 4.8 TB/s).

// the potential around one plane of a block: rows 0, 1 at x = -1 .. 2 (relative
// to the block's cells), rows -1 and 2 at x = 0, 1
template <typename T> struct AccPlane {
    T x[2][4], y[2][2];
};
template <typename T>
__device__ __forceinline__ AccPlane<T> load_acc_plane(const T* __restrict__ f, const unsigned yrow[4], int ex0,
                                                      const int xi[4], bool vload) {
    using V2 = typename Cplx<T>::type;
    AccPlane<T> r;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const T* __restrict__ row = f + yrow[1 + b];
        if (vload) {
            const V2 u = *reinterpret_cast<const V2*>(row + ex0), v = *reinterpret_cast<const V2*>(row + ex0 + 2);
            r.x[b][0] = u.x; r.x[b][1] = u.y; r.x[b][2] = v.x; r.x[b][3] = v.y;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) r.x[b][k] = row[xi[k]];
        }
#pragma unroll
        for (int a = 0; a < 2; ++a) r.y[b][a] = f[yrow[3 * b] + xi[1 + a]];
    }
    return r;
}
// a parent plane's 2x2 values of a field at the block's four (x, y) positions
template <typename T>
__device__ __forceinline__ void lerp_plane(const T* __restrict__ f, unsigned base, int P0, T out[2][2]) {
    const T a = (T)0.75, b = (T)0.25;
    const T q00 = f[base], q01 = f[base + 1], q10 = f[base + P0], q11 = f[base + P0 + 1];
    const T x00 = a * q00 + b * q01, x01 = b * q00 + a * q01, x10 = a * q10 + b * q11, x11 = b * q10 + a * q11;
    out[0][0] = a * x00 + b * x10;
    out[0][1] = a * x01 + b * x11;
    out[1][0] = b * x00 + a * x10;
    out[1][1] = b * x01 + a * x11;
}

// this thread's column of blocks of a marching kernel: blocks [bz0, bz1) at
// output cells ex0, ey0; false: none
struct AccColumn {
    int ex0, ey0, bz0, bz1;
    __device__ __forceinline__ bool start(const GridDev& g, int tile, int zs) {
        const int nbx = g.acc_nb[0], ncol = nbx * g.acc_nb[1];
        const int ncc = (ncol + kAccThreads - 1) / kAccThreads;   // CTAs across the columns
        const int seg = tile / ncc;
        const int col = (tile - seg * ncc) * kAccThreads + (int)threadIdx.x;
        if (col >= ncol) return false;
        const int by = col / nbx;
        ex0 = 2 * (col - by * nbx) - g.acc_sh[0];
        ey0 = 2 * by - g.acc_sh[1];
        bz0 = seg * zs;
        bz1 = min(g.acc_nb[2], bz0 + zs);
        return true;
    }
};
// the parent's phi (0) and accelerations (1-3) along that column: the planes
// below (yp) and above (yn) a block, interpolated in x and y
template <typename T, bool CARRY> struct AccCarry {
    const T* pf[4];
    int P0;
    unsigned P01, pbase;
    T yp[4][2][2], yn[4][2][2];
    __device__ __forceinline__ bool start(const LevelDev& L, const GridDev& g, const GridDev* __restrict__ pgrids,
                                          const void* const* __restrict__ pphi_p,
                                          const void* const* __restrict__ pacc_p, const AccColumn& c) {
        if (!CARRY) return true;
        const GridDev& p = pgrids[g.parent];
        P0 = p.N[0] + 2;
        P01 = (unsigned)P0 * (p.N[1] + 2);
        const unsigned pn = P01 * (p.N[2] + 2);
        pf[0] = reinterpret_cast<const T*>(pphi_p[g.parent]);
#pragma unroll
        for (int j = 0; j < 3; ++j) pf[1 + j] = reinterpret_cast<const T*>(pacc_p[g.parent]) + (size_t)j * pn;
        // parent cell k of the odd level cell (2k+1) of each pair
        const long long kx = ((g.start[0] + c.ex0 - 1) - 1) >> 1, ky = ((g.start[1] + c.ey0 - 1) - 1) >> 1;
        const long long kz = ((g.start[2] + 2 * c.bz0 - g.acc_sh[2] - 1) - 1) >> 1;
        pbase = (unsigned)(kx - p.start[0] + 1) + (unsigned)(ky - p.start[1] + 1) * (unsigned)P0 +
                (unsigned)(kz - p.start[2] + 1) * P01;
        // the blocks' parent cells: pbase .. pbase + 1 + P0 + (bz1 - bz0) P01
        if (!APM_IN_BOUNDS((long long)pbase + 1 + P0 + (long long)(c.bz1 - c.bz0) * P01, pn, L.status)) return false;
#pragma unroll
        for (int j = 0; j < 4; ++j) lerp_plane(pf[j], pbase, P0, yp[j]);
        return true;
    }
    __device__ __forceinline__ void next() {   // the plane above the block
        if (!CARRY) return;
        pbase += P01;
#pragma unroll
        for (int j = 0; j < 4; ++j) lerp_plane(pf[j], pbase, P0, yn[j]);
    }
    // field j of the block's cells (0, b, z), (1, b, z)
    __device__ __forceinline__ void add(int j, int z, int b, T& v0, T& v1) const {
        if (!CARRY) return;
        const T a = z == 0 ? (T)0.75 : (T)0.25, d = z == 0 ? (T)0.25 : (T)0.75;
        v0 += a * yp[j][b][0] + d * yn[j][b][0];
        v1 += a * yp[j][b][1] + d * yn[j][b][1];
    }
    __device__ __forceinline__ void up() {
        if constexpr (CARRY) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int b = 0; b < 2; ++b)
#pragma unroll
                    for (int a = 0; a < 2; ++a) yp[j][b][a] = yn[j][b][a];
        }
    }
};

template <typename T, bool CARRY>
__global__ void __launch_bounds__(kAccThreads, AccMinCtas<T>::march) k_accel(
    LevelDev L, const GridDev* __restrict__ pgrids, const void* const* __restrict__ phis_p,
    const void* const* __restrict__ pphi_p, const void* const* __restrict__ pacc_p, void* const* __restrict__ phi_p,
    void* const* __restrict__ acc_p, const Chunk* __restrict__ chunks, int zs) {
    const unsigned block = begin_kernel();
    const Chunk ch = chunks[block];
    const GridDev& g = L.g[ch.grid];
    AccColumn col;
    if (!col.start(g, ch.tile, zs)) return;
    const int ex0 = col.ex0, ey0 = col.ey0;
    const int E0 = g.N[0] + 2, E1 = g.N[1] + 2, E2 = g.N[2] + 2;
    const unsigned ncell = (unsigned)E0 * E1 * E2;
    const int W0 = g.W[0], W1 = g.W[1], W2 = g.W[2];
    const T* __restrict__ phis = reinterpret_cast<const T*>(phis_p[ch.grid]);
    T* __restrict__ phi = reinterpret_cast<T*>(phi_p[ch.grid]);
    T* __restrict__ acc = reinterpret_cast<T*>(acc_p[ch.grid]);
    const T inv2d = (T)g.inv2d;
    // output cell e has phis index e + 1 on each axis; clamped into [0, W)
    const unsigned sz = (unsigned)W0 * W1;
    unsigned yrow[4];
    int xi[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        yrow[k] = (unsigned)W0 * (unsigned)min(max(ey0 + k, 0), W1 - 1);
        xi[k] = min(max(ex0 + k, 0), W0 - 1);
    }
    // pair loads and stores need even row lengths and pointers aligned to two elements
    using V2 = typename Cplx<T>::type;
    const size_t amask = 2 * sizeof(T) - 1;
    const bool vpair = !((W0 | E0 | ex0) & 1) && !(reinterpret_cast<size_t>(phis) & amask) &&
                       !(reinterpret_cast<size_t>(phi) & amask) && !(reinterpret_cast<size_t>(acc) & amask) &&
                       !((size_t)ncell & 1);
    const bool vload = vpair && ex0 >= 0 && ex0 + 3 <= W0 - 1;
    // cells written: x = ex0 + a, y = ey0 + b
    const bool wx0 = ex0 >= 0 && ex0 < E0, wx1 = ex0 + 1 < E0;
    const bool wy0 = ey0 >= 0 && ey0 < E1, wy1 = ey0 + 1 < E1;
    AccCarry<T, CARRY> carry;
    if (!carry.start(L, g, pgrids, pphi_p, pacc_p, col)) return;
    auto plane = [&](int k) { return phis + sz * (unsigned)min(max(k, 0), W2 - 1); };
    int ez0 = 2 * col.bz0 - g.acc_sh[2];
    T z0[2][2];   // centres of the plane below the block
    {
        const T* __restrict__ f = plane(ez0);
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) z0[b][a] = f[yrow[1 + b] + xi[1 + a]];
    }
    AccPlane<T> p1 = load_acc_plane(plane(ez0 + 1), yrow, ex0, xi, vload);
#pragma unroll 1
    for (int bz = col.bz0; bz < col.bz1; ++bz, ez0 += 2) {
        const AccPlane<T> p2 = load_acc_plane(plane(ez0 + 2), yrow, ex0, xi, vload);
        const AccPlane<T> p3 = load_acc_plane(plane(ez0 + 3), yrow, ex0, xi, vload);
        carry.next();
        const bool wz[2] = {ez0 >= 0 && ez0 < E2, ez0 + 1 < E2};
        // field j (0 phi, 1-3 acc) of cells (.., b, c): values v0, v1 plus the carry
        auto put = [&](T* __restrict__ f, int j, int c, int b, T v0, T v1) {
            carry.add(j, c, b, v0, v1);
            if (!((b == 0 ? wy0 : wy1) && wz[c])) return;
            // signed: with ex0 = -1 the row's first written cell is o[1] (fields hold fewer than 2^31 cells)
            T* __restrict__ o = f + (ex0 + E0 * ((ey0 + b) + E1 * (ez0 + c)));
            if (vpair && wx0 && wx1) {
                *reinterpret_cast<V2*>(o) = mk2(v0, v1);
            } else {
                if (wx0) o[0] = v0;
                if (wx1) o[1] = v1;
            }
        };
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const AccPlane<T>& p = c == 0 ? p1 : p2;
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                put(phi, 0, c, b, p.x[b][1], p.x[b][2]);
                put(acc, 1, c, b, -(p.x[b][2] - p.x[b][0]) * inv2d, -(p.x[b][3] - p.x[b][1]) * inv2d);
                T gy[2], gz[2];
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const T ylo = b == 0 ? p.y[0][a] : p.x[0][1 + a], yhi = b == 0 ? p.x[1][1 + a] : p.y[1][a];
                    const T zlo = c == 0 ? z0[b][a] : p1.x[b][1 + a], zhi = c == 0 ? p2.x[b][1 + a] : p3.x[b][1 + a];
                    gy[a] = -(yhi - ylo) * inv2d;
                    gz[a] = -(zhi - zlo) * inv2d;
                }
                put(acc + ncell, 2, c, b, gy[0], gy[1]);
                put(acc + 2 * ncell, 3, c, b, gz[0], gz[1]);
            }
        }
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) z0[b][a] = p2.x[b][1 + a];
        carry.up();
        p1 = p3;
    }
}


// index of the grid of level L whose interior holds level cell ic, or -1
__device__ int find_owner(const LevelDev& L, const long long ic[3]) {
    if (L.is_root) {
        const GridDev& g = L.g[0];
        for (int j = 0; j < 3; ++j)
            if (ic[j] < 0 || ic[j] >= g.N[j]) return -1;
        return 0;
    }
    const TileMap& m = L.map;
    long long t[3];
    for (int j = 0; j < 3; ++j) {
        long long rel = ic[j] - m.lo[j];
        if (rel < 0) return -1;
        t[j] = rel >> m.shift;
        if (t[j] >= m.nt[j]) return -1;
    }
    long long tile = t[0] + (long long)m.nt[0] * (t[1] + (long long)m.nt[1] * t[2]);
    for (int e = m.own_off[tile]; e < m.own_off[tile + 1]; ++e) {
        int gi = m.own_list[e];
        const GridDev& g = L.g[gi];
        bool in = true;
        for (int j = 0; j < 3; ++j)
            if (ic[j] < g.start[j] || ic[j] >= g.start[j] + g.N[j]) in = false;
        if (in) return gi;
    }
    return -1;
}

// The 27 interpolation weights of a particle at fixed-point position X on a
// level with `fb` fraction bits.  FP64: the deposit's fixed-point weights
// exactly (outer products ((wx wy) wz) rounded on the scale 2^63, the centre one
// minus their sum).  FP32: the same TSC weights evaluated in FP32 from the
// offsets (t = f 2^-fb; (1-t)^2/2, 3/4 - (t-1/2)^2, t^2/2; products (wx wy) wz),
// within a few FP32 roundings of the fixed-point ones.
template <typename T> struct InterpWeights;
template <> struct InterpWeights<double> {
    double wq[3][3][3];
    __device__ __forceinline__ InterpWeights(const long long X[3], int fb) {
        unsigned long long w[3][3];
        for (int j = 0; j < 3; ++j) tsc_fixed(X[j], fb, w[j]);
        unsigned long long wsum = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int b = 0; b < 3; ++b)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (a == 1 && b == 1 && c == 1) continue;
                    const unsigned long long q = wmul63(wmul63(w[0][a], w[1][b]), w[2][c]);
                    wsum += q;
                    wq[c][b][a] = __ull2double_rn(q) * 1.0842021724855044e-19;   // 2^-63
                }
        wq[1][1][1] = __ull2double_rn(kOne63 - wsum) * 1.0842021724855044e-19;
    }
    __device__ __forceinline__ double operator()(int c, int b, int a) const { return wq[c][b][a]; }
};
// The products are formed where they are used: 9 registers across the loads, not 27
// (1 M random particles on 63^3 212 -> 201 us, 4.2 M in bin order on 256^3 593 -> 576;
// 904 -> 908 for 16.8 M lattice ones on 512^3).
template <> struct InterpWeights<float> {
    float w[3][3];
    __device__ __forceinline__ InterpWeights(const long long X[3], int fb) {
        const float sc = __int_as_float((127 - fb) << 23);   // 2^-fb
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const long long i = X[j] >> fb;
            const float t = __uint2float_rn((unsigned)(X[j] - (i << fb))) * sc;   // offset < 2^fb <= 2^31
            const float u = 1.0f - t;
            w[j][0] = 0.5f * u * u;
            w[j][2] = 0.5f * t * t;
            w[j][1] = 0.75f - (t - 0.5f) * (t - 0.5f);
        }
    }
    __device__ __forceinline__ float operator()(int c, int b, int a) const { return w[0][a] * (w[1][b] * w[2][c]); }
};

// TSC interpolation of the cell accelerations A (3 x (N+2)^3 of grid g, level L)
// at fixed-point position X; writes out[p], out[n + p], out[2n + p].
template <typename T>
__device__ __forceinline__ void interp_from(const LevelDev& L, const GridDev& g, const T* __restrict__ A,
                                            const long long X[3], long long p, long long n,
                                            T* __restrict__ out) {
    const InterpWeights<T> wq(X, L.frac_bits);
    const int E0 = g.N[0] + 2, E1 = g.N[1] + 2;
    const unsigned ncell = (unsigned)E0 * E1 * (g.N[2] + 2);
    const bool fold = g.mode == 1;
    int lc[3];
    for (int j = 0; j < 3; ++j) lc[j] = (int)((X[j] >> L.frac_bits) - g.start[j]);
    // the owner's interior holds the particle's cell (fold: the root's box)
    for (int j = 0; j < 3; ++j)
        if (!APM_IN_BOUNDS(fold ? min(max(lc[j], 0), g.N[j] - 1) : lc[j], g.N[j], L.status)) return;
    T a0 = 0, a1 = 0, a2 = 0;
    // the three cells of a row lie in two aligned pairs: 54 pair loads instead of
    // 81 (the load/store unit is what bounds the kernel: 72% of its peak with
    // single loads on the lattice).  Rows and components of even length from an
    // aligned pointer start on a pair, so the pairs stay inside the row (its
    // first cell has the parity of lc[0]); a cloud folded at an isolated root's
    // faces is not contiguous.  The same bits; a Plummer sphere of 1 M 182 -> 155
    // us in bin order and 236 -> 186 in its own, 16.8 M lattice particles 889 ->
    // 875.  (The deposit's arrangement, 8 particles' rows a load, took 154 us
    // for the sphere in its own order, but 1040 for the lattice, whose
    // neighbouring lanes share sectors already.)
    using V2 = typename Cplx<T>::type;
    bool pairs = !(E0 & 1) && !(ncell & 1) && !(reinterpret_cast<size_t>(A) & (2 * sizeof(T) - 1));
    for (int j = 0; j < 3; ++j) pairs = pairs && (!fold || (lc[j] > 0 && lc[j] < g.N[j] - 1));
    if (pairs) {
        const bool odd = lc[0] & 1;
        const T* __restrict__ base =
            A + ((unsigned)(lc[0] & ~1) + (unsigned)E0 * ((unsigned)lc[1] + (unsigned)E1 * (unsigned)lc[2]));
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const unsigned row = (unsigned)E0 * ((unsigned)b + (unsigned)E1 * (unsigned)c);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const V2* __restrict__ q = reinterpret_cast<const V2*>(base + (row + (unsigned)j * ncell));
                    const V2 u = q[0], v = q[1];
                    T& acc = j == 0 ? a0 : (j == 1 ? a1 : a2);
                    acc += wq(c, b, 0) * (odd ? u.y : u.x);
                    acc += wq(c, b, 1) * (odd ? v.x : u.y);
                    acc += wq(c, b, 2) * (odd ? v.y : v.x);
                }
            }
        out[p] = a0;
        out[n + p] = a1;
        out[2 * n + p] = a2;
        return;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int z = lc[2] + c - 1;
        if (fold) z = z < 0 ? 0 : (z >= g.N[2] ? g.N[2] - 1 : z);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            int y = lc[1] + b - 1;
            if (fold) y = y < 0 ? 0 : (y >= g.N[1] ? g.N[1] - 1 : y);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                int x = lc[0] + a - 1;
                if (fold) x = x < 0 ? 0 : (x >= g.N[0] ? g.N[0] - 1 : x);
                const T wt = wq(c, b, a);
                unsigned idx = (unsigned)(x + 1) + (unsigned)E0 * ((unsigned)(y + 1) + (unsigned)E1 * (unsigned)(z + 1));
                a0 += wt * A[idx];
                a1 += wt * A[ncell + idx];
                a2 += wt * A[2 * ncell + idx];
            }
        }
    }
    out[p] = a0;
    out[n + p] = a1;
    out[2 * n + p] = a2;
}

template <typename T>
__device__ __forceinline__ void particle_position(const LevelDev& L, const Particles& P, long long p,
                                                  double half_dt, long long X[3]) {
    constexpr bool kBits = sizeof(T) == 8;
    X[0] = fixed_position<kBits>(drift_raw(P.x[p], P.vx[p], half_dt), L);
    X[1] = fixed_position<kBits>(drift_raw(P.y[p], P.vy[p], half_dt), L);
    X[2] = fixed_position<kBits>(drift_raw(P.z[p], P.vz[p], half_dt), L);
}

// One level: the particles owned by a grid of L and by no grid of the finer
// level F (the finest grid holding a particle supplies its acceleration).
template <typename T>
__global__ void __launch_bounds__(256) k_interp(LevelDev L, LevelDev F, int has_finer, Particles P,
                                                double half_dt, const void* const* __restrict__ acc_p,
                                                T* __restrict__ out) {
    const unsigned block = begin_kernel();
    const long long i = (long long)block * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const long long p = P.at(i);
    long long X[3];
    particle_position<T>(L, P, p, half_dt, X);
    long long ic[3];
    for (int j = 0; j < 3; ++j) ic[j] = X[j] >> L.frac_bits;
    int gi = find_owner(L, ic);
    if (gi < 0) return;
    if (has_finer) {
        long long fc[3];
        for (int j = 0; j < 3; ++j) fc[j] = X[j] >> F.frac_bits;
        if (find_owner(F, fc) >= 0) return;
    }
    interp_from<T>(L, L.g[gi], reinterpret_cast<const T*>(acc_p[gi]), X, p, P.n, out);
}

// Every level in one pass: each particle's position is converted once and its
// owner searched from the root down (a finer owner lies inside a coarser one);
// the finest owner supplies the acceleration.  accs[l]: the acceleration
// pointer table of level l.
// CTA size and minimum resident CTAs per SM of the all-level interpolation
#ifndef APM_INT_THREADS
#define APM_INT_THREADS 128
#endif
#ifndef APM_INT_MIN_CTAS
#define APM_INT_MIN_CTAS 8
#endif
constexpr int kIntThreads = APM_INT_THREADS;

template <typename T>
__global__ void __launch_bounds__(kIntThreads, APM_INT_MIN_CTAS) k_interp_levels(const LevelDev* __restrict__ levels, int nl, Particles P,
                                                       double half_dt, const void* const* const* __restrict__ accs,
                                                       T* __restrict__ out) {
    const unsigned block = begin_kernel();
    const long long i = (long long)block * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const long long p = P.at(i);
    long long X[3];
    particle_position<T>(levels[0], P, p, half_dt, X);
    int own_l = -1, own_g = -1;
    for (int l = 0; l < nl; ++l) {
        long long ic[3];
        for (int j = 0; j < 3; ++j) ic[j] = X[j] >> levels[l].frac_bits;
        const int gi = find_owner(levels[l], ic);
        if (gi < 0) break;
        own_l = l;
        own_g = gi;
    }
    if (own_l < 0) return;
    const LevelDev& L = levels[own_l];
    interp_from<T>(L, L.g[own_g], reinterpret_cast<const T*>(accs[own_l][own_g]), X, p, P.n, out);
}

// The spectral gradient's accelerations: phi and acc_j are the solve's four
// windows of [-2, N+2) plus the parent's, on k_accel's columns of blocks; each
// thread marches up z and keeps the parent plane between two blocks, so a block
// loads 16 parent values instead of 32.  8 grids of 100^3: 113 -> 68 us.
template <typename T, bool CARRY>
__global__ void __launch_bounds__(kAccThreads, AccMinCtas<T>::march) k_accel_spectral(
    LevelDev L, const GridDev* __restrict__ pgrids, const void* const* __restrict__ phis_p,
    const void* const* __restrict__ pphi_p, const void* const* __restrict__ pacc_p, void* const* __restrict__ phi_p,
    void* const* __restrict__ acc_p, const Chunk* __restrict__ chunks, int zs) {
    const unsigned block = begin_kernel();
    const Chunk ch = chunks[block];
    const GridDev& g = L.g[ch.grid];
    AccColumn c;
    if (!c.start(g, ch.tile, zs)) return;
    const int E0 = g.N[0] + 2, E1 = g.N[1] + 2, E2 = g.N[2] + 2;
    const unsigned ncell = (unsigned)E0 * E1 * E2;
    const int W0 = g.W[0], W1 = g.W[1];
    const unsigned sz = (unsigned)W0 * W1, nw = sz * (unsigned)g.W[2];
    const T* __restrict__ phis = reinterpret_cast<const T*>(phis_p[ch.grid]);
    T* __restrict__ phi = reinterpret_cast<T*>(phi_p[ch.grid]);
    T* __restrict__ acc = reinterpret_cast<T*>(acc_p[ch.grid]);
    using V2 = typename Cplx<T>::type;
    const size_t amask = 2 * sizeof(T) - 1;
    const bool vst = !((E0 | c.ex0) & 1) && !(reinterpret_cast<size_t>(phi) & amask) &&
                     !(reinterpret_cast<size_t>(acc) & amask) && !(ncell & 1);
    // output cell e is window cell e + 1 on each axis
    const bool wx0 = c.ex0 >= 0 && c.ex0 < E0, wx1 = c.ex0 + 1 < E0;
    const bool vld = !((W0 | nw) & 1) && (c.ex0 & 1) && wx0 && wx1 && !(reinterpret_cast<size_t>(phis) & amask);
    AccCarry<T, CARRY> carry;
    if (!carry.start(L, g, pgrids, pphi_p, pacc_p, c)) return;
    int ez0 = 2 * c.bz0 - g.acc_sh[2];
#pragma unroll 1
    for (int bz = c.bz0; bz < c.bz1; ++bz, ez0 += 2) {
        T v[4][2][2][2];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int z = 0; z < 2; ++z)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int ey = c.ey0 + b, ez = ez0 + z;
                    const bool ok = ey >= 0 && ey < E1 && ez >= 0 && ez < E2;
                    const T* __restrict__ q = phis + ((size_t)j * nw + (unsigned)(W0 * (ey + 1)) + sz * (unsigned)(ez + 1));
                    if (vld) {
                        const V2 u = ok ? *reinterpret_cast<const V2*>(q + c.ex0 + 1) : mk2((T)0, (T)0);
                        v[j][z][b][0] = u.x;
                        v[j][z][b][1] = u.y;
                    } else {
                        v[j][z][b][0] = ok && wx0 ? q[c.ex0 + 1] : (T)0;
                        v[j][z][b][1] = ok && wx1 ? q[c.ex0 + 2] : (T)0;
                    }
                }
        carry.next();
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int z = 0; z < 2; ++z)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int ey = c.ey0 + b, ez = ez0 + z;
                    if (!(ey >= 0 && ey < E1 && ez >= 0 && ez < E2)) continue;
                    T v0 = v[j][z][b][0], v1 = v[j][z][b][1];
                    carry.add(j, z, b, v0, v1);
                    T* __restrict__ o = (j == 0 ? phi : acc + (size_t)(j - 1) * ncell) + (c.ex0 + E0 * (ey + E1 * ez));
                    if (vst && wx0 && wx1) {
                        *reinterpret_cast<V2*>(o) = mk2(v0, v1);
                    } else {
                        if (wx0) o[0] = v0;
                        if (wx1) o[1] = v1;
                    }
                }
        carry.up();
    }
}

// The four-point gradient (Sec. 2.2; apm_gradient), one 2x2x2 block of k_accel's
// per thread (flat ranges of blocks, the same parent interpolation):
//   phi(c)   = phis(c) + I(parent phi)(c)
//   acc_j(c) = A_j(c) + I(parent acc_j)(c),        c in [-1, N]^3, with
//   A_j = -(8 (phis(c+e_j) - phis(c-e_j)) - (phis(c+2e_j) - phis(c-2e_j))) / (12 delta)
//         (phis spans [-3, N+3)).
// Output cell e (index 0..E-1) is level cell e - 1 and phis cell e - 1 + h.
template <typename T>
__global__ void __launch_bounds__(kAccThreads, AccMinCtas<T>::value) k_accel_var(
    LevelDev L, const GridDev* __restrict__ pgrids, const void* const* __restrict__ phis_p,
    const void* const* __restrict__ pphi_p, const void* const* __restrict__ pacc_p,
    void* const* __restrict__ phi_p, void* const* __restrict__ acc_p, const Chunk* __restrict__ chunks) {
    const unsigned block = begin_kernel();
    const Chunk ch = chunks[block];
    const GridDev& g = L.g[ch.grid];
    const int E0 = g.N[0] + 2, E1 = g.N[1] + 2, E2 = g.N[2] + 2;
    const unsigned ncell = (unsigned)E0 * E1 * E2;
    const int h = g.h;
    const unsigned W0 = g.W[0], W01 = (unsigned)g.W[0] * g.W[1];
    const unsigned nw = W01 * (unsigned)g.W[2];
    const int nbx = g.acc_nb[0], nby = g.acc_nb[1];
    const int nbrows = nby * g.acc_nb[2];
    const T* __restrict__ phis = reinterpret_cast<const T*>(phis_p[ch.grid]);
    T* __restrict__ phi = reinterpret_cast<T*>(phi_p[ch.grid]);
    T* __restrict__ acc = reinterpret_cast<T*>(acc_p[ch.grid]);
    const bool carry = pphi_p != nullptr && g.parent >= 0;
    const T* __restrict__ pphi = carry ? reinterpret_cast<const T*>(pphi_p[g.parent]) : nullptr;
    const T* __restrict__ pacc = carry ? reinterpret_cast<const T*>(pacc_p[g.parent]) : nullptr;
    int P0 = 0;
    unsigned P01 = 0, pn = 0;
    long long ps[3] = {0, 0, 0};
    if (carry) {
        const GridDev& p = pgrids[g.parent];
        P0 = p.N[0] + 2;
        P01 = (unsigned)P0 * (p.N[1] + 2);
        pn = P01 * (p.N[2] + 2);
        ps[0] = p.start[0]; ps[1] = p.start[1]; ps[2] = p.start[2];
    }
    const T inv12d = (T)g.inv12d;
    const unsigned st[3] = {1u, W0, W01};
    // two-element accesses need even row lengths and pointers aligned to two elements
    using V2 = typename Cplx<T>::type;
    const size_t amask = 2 * sizeof(T) - 1;
    const bool vout = !(E0 & 1) && !(ncell & 1) && !(reinterpret_cast<size_t>(phi) & amask) &&
                      !(reinterpret_cast<size_t>(acc) & amask);
    const bool vin = !(W0 & 1) && !(W01 & 1) && !(nw & 1) && !(reinterpret_cast<size_t>(phis) & amask);
    const long long nblocks = (long long)nbx * nbrows;
    const long long f0 = (long long)ch.tile * kAccBlocksPerCta;
    const int count = (int)min((long long)kAccBlocksPerCta, nblocks - f0);
    int last = -1;
    int ey0 = 0, ez0 = 0;
    unsigned prow = 0;
    for (FlatWalk it(f0, count, nbx); it.ok(); it.next()) {
        if (it.r != last) {
            last = it.r;
            const int by = it.r % nby, bz = it.r / nby;
            ey0 = 2 * by - g.acc_sh[1];
            ez0 = 2 * bz - g.acc_sh[2];
            if (carry) {
                const long long ky = ((g.start[1] + ey0 - 1) - 1) >> 1;
                const long long kz = ((g.start[2] + ez0 - 1) - 1) >> 1;
                prow = (unsigned)(ky - ps[1] + 1) * (unsigned)P0 + (unsigned)(kz - ps[2] + 1) * P01;
            }
        }
        const int ex0 = 2 * it.x - g.acc_sh[0];
        unsigned pbase = 0;
        if (carry) {
            const long long kx = ((g.start[0] + ex0 - 1) - 1) >> 1;
            pbase = prow + (unsigned)(kx - ps[0] + 1);
            if (!APM_IN_BOUNDS((long long)pbase + 1 + P0 + P01, pn, L.status)) continue;
        }
        bool wr[2][2][2];
        unsigned o[2][2][2], c0[2][2][2];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const int ex = ex0 + a, ey = ey0 + b, ez = ez0 + c;
                    wr[c][b][a] = ex >= 0 && ex < E0 && ey >= 0 && ey < E1 && ez >= 0 && ez < E2;
                    o[c][b][a] = (unsigned)ex + (unsigned)E0 * ((unsigned)ey + (unsigned)E1 * (unsigned)ez);
                    c0[c][b][a] = (unsigned)(ex - 1 + h) + W0 * (unsigned)(ey - 1 + h) + W01 * (unsigned)(ez - 1 + h);
                }
        // a row pair (a = 0, 1) with both cells written moves as two-element
        // loads and stores where aligned; other pairs cell by cell
        const bool pst = vout && !(ex0 & 1);               // o[.][.][0] even
        const bool pld = vin && !(c0[0][0][0] & 1);        // c0[.][.][0] even (W0, W01 even)
        T out[2][2][2], q[2][2][2];
        if (carry) {
            load_parent<T>(pphi, pbase, P0, P01, q);
            lerp_block<T>(q, out);
        }
        auto put = [&](T* __restrict__ f, unsigned i, int c, int b, T v0, T v1) {
            if (pst && wr[c][b][0] && wr[c][b][1]) {
                *reinterpret_cast<V2*>(f + i) = mk2(v0, v1);
            } else {
                if (wr[c][b][0]) f[i] = v0;
                if (wr[c][b][1]) f[i + 1] = v1;
            }
        };
        auto ld2 = [&](const T* __restrict__ f, unsigned i, T& v0, T& v1) {
            if (pld) {
                const V2 u = *reinterpret_cast<const V2*>(f + i);
                v0 = u.x;
                v1 = u.y;
            } else {
                v0 = f[i];
                v1 = f[i + 1];
            }
        };
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const unsigned ci = c0[c][b][0];
                T v0 = 0, v1 = 0;
                if (wr[c][b][0] && wr[c][b][1]) {
                    ld2(phis, ci, v0, v1);
                } else {
                    if (wr[c][b][0]) v0 = phis[ci];
                    if (wr[c][b][1]) v1 = phis[ci + 1];
                }
                if (carry) {
                    v0 += out[c][b][0];
                    v1 += out[c][b][1];
                }
                put(phi, o[c][b][0], c, b, v0, v1);
            }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (carry) {
                load_parent<T>(pacc + j * pn, pbase, P0, P01, q);
                lerp_block<T>(q, out);
            }
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const unsigned ci = c0[c][b][0];
                    T v[2] = {0, 0};
                    if (wr[c][b][0] && wr[c][b][1]) {
                        if (j == 0) {   // x: cells ci-2 .. ci+3
                            T m2, m1, p0, p1, p2, p3;
                            ld2(phis, ci - 2, m2, m1);
                            ld2(phis, ci, p0, p1);
                            ld2(phis, ci + 2, p2, p3);
                            v[0] = -((T)8 * (p1 - m1) - (p2 - m2)) * inv12d;
                            v[1] = -((T)8 * (p2 - p0) - (p3 - m1)) * inv12d;
                        } else {
                            T a1[2], b1[2], a2[2], b2[2];
                            ld2(phis, ci + st[j], a1[0], a1[1]);
                            ld2(phis, ci - st[j], b1[0], b1[1]);
                            ld2(phis, ci + 2 * st[j], a2[0], a2[1]);
                            ld2(phis, ci - 2 * st[j], b2[0], b2[1]);
#pragma unroll
                            for (int a = 0; a < 2; ++a)
                                v[a] = -((T)8 * (a1[a] - b1[a]) - (a2[a] - b2[a])) * inv12d;
                        }
                    } else {
#pragma unroll
                        for (int a = 0; a < 2; ++a) {
                            if (!wr[c][b][a]) continue;
                            const unsigned cc = ci + a;
                            const T d1 = phis[cc + st[j]] - phis[cc - st[j]];
                            const T d2 = phis[cc + 2 * st[j]] - phis[cc - 2 * st[j]];
                            v[a] = -((T)8 * d1 - d2) * inv12d;
                        }
                    }
                    if (carry) {
                        v[0] += out[c][b][0];
                        v[1] += out[c][b][1];
                    }
                    put(acc + j * ncell, o[c][b][0], c, b, v[0], v[1]);
                }
        }
    }
}

}  // namespace

template <typename T>
cudaError_t launch_accel(const LevelDev& L, const GridDev* parent_grids, const void* const* phis,
                         const void* const* pphi, const void* const* pacc, void* const* phi,
                         void* const* acc, const Chunk* chunks, int n_chunks, int zs,
                         cudaStream_t s) {
    if (n_chunks <= 0) return cudaSuccess;
    if (pphi)   // every grid of a level that gets parent fields has a parent
        return launch_kernel(k_accel<T, true>, n_chunks, kAccThreads, 0, s, L, parent_grids, phis, pphi, pacc, phi,
                             acc, chunks, zs);
    else
        return launch_kernel(k_accel<T, false>, n_chunks, kAccThreads, 0, s, L, parent_grids, phis, pphi, pacc,
                             phi, acc, chunks, zs);
}

template <typename T>
cudaError_t launch_accel_var(const LevelDev& L, const GridDev* parent_grids, const void* const* phis,
                               const void* const* pphi, const void* const* pacc, void* const* phi,
                               void* const* acc, const Chunk* chunks, int n_chunks, int grad, int zs,
                               cudaStream_t s) {
    if (n_chunks <= 0) return cudaSuccess;
    if (grad == APM_GRAD_FD4)
        return launch_kernel(k_accel_var<T>, n_chunks, kAccThreads, 0, s, L, parent_grids, phis, pphi, pacc, phi, acc,
                             chunks);
    return pphi ? launch_kernel(k_accel_spectral<T, true>, n_chunks, kAccThreads, 0, s, L, parent_grids, phis, pphi,
                                pacc, phi, acc, chunks, zs)
                : launch_kernel(k_accel_spectral<T, false>, n_chunks, kAccThreads, 0, s, L, parent_grids, phis, pphi,
                                pacc, phi, acc, chunks, zs);
}

template <typename T>
cudaError_t launch_interp(const LevelDev& L, const LevelDev* finer, const Particles& P,
                          double half_dt, const void* const* acc, void* out, cudaStream_t s) {
    if (P.n <= 0) return cudaSuccess;
    unsigned blocks = (unsigned)((P.n + 255) / 256);
    LevelDev F = finer ? *finer : L;
    return launch_kernel(k_interp<T>, blocks, 256, 0, s, L, F, finer ? 1 : 0, P, half_dt, acc,
                         reinterpret_cast<T*>(out));
}

template <typename T>
cudaError_t launch_interp_levels(const LevelDev* levels, int nl, const Particles& P, double half_dt,
                                 const void* const* const* accs, void* out, cudaStream_t s) {
    if (P.n <= 0 || nl <= 0) return cudaSuccess;
    unsigned blocks = (unsigned)((P.n + kIntThreads - 1) / kIntThreads);
    return launch_kernel(k_interp_levels<T>, blocks, kIntThreads, 0, s, levels, nl, P, half_dt, accs,
                         reinterpret_cast<T*>(out));
}

template cudaError_t launch_accel<float>(const LevelDev&, const GridDev*, const void* const*,
                                         const void* const*, const void* const*, void* const*,
                                         void* const*, const Chunk*, int, int, cudaStream_t);
template cudaError_t launch_accel<double>(const LevelDev&, const GridDev*, const void* const*,
                                          const void* const*, const void* const*, void* const*,
                                          void* const*, const Chunk*, int, int, cudaStream_t);
template cudaError_t launch_accel_var<float>(const LevelDev&, const GridDev*, const void* const*,
                                               const void* const*, const void* const*, void* const*,
                                               void* const*, const Chunk*, int, int, int, cudaStream_t);
template cudaError_t launch_accel_var<double>(const LevelDev&, const GridDev*, const void* const*,
                                                const void* const*, const void* const*, void* const*,
                                                void* const*, const Chunk*, int, int, int, cudaStream_t);
template cudaError_t launch_interp<float>(const LevelDev&, const LevelDev*, const Particles&, double,
                                          const void* const*, void*, cudaStream_t);
template cudaError_t launch_interp<double>(const LevelDev&, const LevelDev*, const Particles&, double,
                                           const void* const*, void*, cudaStream_t);
template cudaError_t launch_interp_levels<float>(const LevelDev*, int, const Particles&, double,
                                                 const void* const* const*, void*, cudaStream_t);
template cudaError_t launch_interp_levels<double>(const LevelDev*, int, const Particles&, double,
                                                  const void* const* const*, void*, cudaStream_t);

}  // namespace apm
