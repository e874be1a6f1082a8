// k_order.cu -- a spatially coherent processing order of the particles: a
// counting sort of the particle indices by the root-level bin (cubes of 2^shift
// root cells) of their drifted positions.  The interpolation kernels then visit
// the particles bin by bin, so a warp's clouds overlap and its gathers touch
// the same cache lines.  The order changes no result: each particle is
// interpolated on its own.
#include <cmath>

#include "apm_internal.cuh"

namespace apm {
namespace {

constexpr int kScanChunk = 2048;   // bins per CTA of the local scan (1024 threads x 2)

// The bin of a particle needs no exact position (any order gives the same
// results), and the FP64 pipe (2 lanes per clock and SM) would bound the pass:
// coordinates and velocities are taken as FP32, in units of 2^ex and 2^ev near
// the box and the box per drift time, by shifting their bits.
struct BinScale {
    int ex, ev;              // exponents of the units
    float cx, cv;            // bins per unit of x, and of v drifted
    float period, inv_period;   // bins per box (periodic root; 0: isolated)
    int nb;
};

// x 2^-ex truncated to FP32 (0 below 2^-126, 2^127 above it or not finite)
__device__ __forceinline__ float float_of(double x, int ex) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int h = (int)(hi & 0x7fffffffu) - (896 + ex) * (1 << 20);
    const unsigned m = h < (1 << 20) ? 0u : (h >= (254 << 20) ? 254u << 23 : __funnelshift_l(lo, (unsigned)h, 3));
    return __uint_as_float(m | (hi & 0x80000000u));
}
__device__ __forceinline__ int bin_of(double x, double v, const BinScale& s) {
    float b = float_of(x, s.ex) * s.cx + float_of(v, s.ev) * s.cv;
    if (s.period > 0.f) b -= s.period * floorf(b * s.inv_period);
    return (int)fminf(fmaxf(b, 0.f), (float)(s.nb - 1));   // NaN: bin 0
}

// bin of each particle and its rank inside the bin (the count before it); the
// lanes of a warp with the same bin share one atomic addition (4.2 M random
// particles, 262144 bins: the whole ordering 154 -> 118 us; a Plummer sphere
// of 1 M, whose core bins hold up to 1e5 particles, 141 -> 94)
__global__ void __launch_bounds__(256) k_order_bins(Particles P, BinScale s, unsigned* __restrict__ count,
                                                    unsigned* __restrict__ key, unsigned* __restrict__ rank) {
    const unsigned block = begin_kernel();
    const long long p = (long long)block * blockDim.x + threadIdx.x;
    const bool live = p < P.n;
    unsigned k = 0xffffffffu;
    if (live) {
        const int bx = bin_of(P.x[p], P.vx[p], s), by = bin_of(P.y[p], P.vy[p], s), bz = bin_of(P.z[p], P.vz[p], s);
        k = (unsigned)(bx + s.nb * (by + s.nb * bz));
    }
    const unsigned same = __match_any_sync(0xffffffffu, k);
    const int lane = threadIdx.x & 31, first = __ffs(same) - 1;
    unsigned base = 0;
    if (live && lane == first) base = atomicAdd(count + k, (unsigned)__popc(same));
    base = __shfl_sync(0xffffffffu, base, first);
    if (live) {
        key[p] = k;
        rank[p] = base + __popc(same & ((1u << lane) - 1u));
    }
}

// exclusive scan of each chunk of kScanChunk counts in place; the chunk's total
// to sums[chunk]
__global__ void __launch_bounds__(1024) k_order_scan_local(unsigned* __restrict__ count, int nbins,
                                                           unsigned* __restrict__ sums) {
    const unsigned block = begin_kernel();
    __shared__ unsigned warp_tot[32];
    const int base = block * kScanChunk + 2 * threadIdx.x;
    const unsigned a = base < nbins ? count[base] : 0u;
    const unsigned b = base + 1 < nbins ? count[base + 1] : 0u;
    const unsigned t = a + b;
    // inclusive scan of t over the CTA: warp shuffles, then the warp totals
    unsigned v = t;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += u;
    }
    if (lane == 31) warp_tot[warp] = v;
    __syncthreads();
    if (warp == 0) {
        unsigned w = warp_tot[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += u;
        }
        warp_tot[lane] = w;   // inclusive over warps
    }
    __syncthreads();
    const unsigned before = v - t + (warp > 0 ? warp_tot[warp - 1] : 0u);   // exclusive prefix of a
    if (base < nbins) count[base] = before;
    if (base + 1 < nbins) count[base + 1] = before + a;
    if (threadIdx.x == blockDim.x - 1) sums[block] = before + t;
}

// exclusive scan of the chunk totals (at most 1024 chunks) in place, one CTA
__global__ void __launch_bounds__(1024) k_order_scan_sums(unsigned* __restrict__ sums, int n) {
    const unsigned block = begin_kernel();   // 0: its address keeps the load behind the wait
    __shared__ unsigned warp_tot[32];
    const unsigned i = block * blockDim.x + threadIdx.x;
    const unsigned t = i < (unsigned)n ? sums[i] : 0u;
    unsigned v = t;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += u;
    }
    if (lane == 31) warp_tot[warp] = v;
    __syncthreads();
    if (warp == 0) {
        unsigned w = warp_tot[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += u;
        }
        warp_tot[lane] = w;
    }
    __syncthreads();
    if (i < (unsigned)n) sums[i] = v - t + (warp > 0 ? warp_tot[warp - 1] : 0u);
}

// perm[slot] = p with slot = (chunk offset + bin offset + rank)
__global__ void __launch_bounds__(256) k_order_scatter(long long n, const unsigned* __restrict__ key,
                                                       const unsigned* __restrict__ rank,
                                                       const unsigned* __restrict__ count,
                                                       const unsigned* __restrict__ sums, int* __restrict__ perm) {
    const unsigned block = begin_kernel();
    const long long p = (long long)block * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const unsigned k = key[p];
    const unsigned slot = sums[k / kScanChunk] + count[k] + rank[p];
    perm[slot] = (int)p;
}

}  // namespace

int order_scan_chunks(int nbins) { return (nbins + kScanChunk - 1) / kScanChunk; }

// bins of 2^shift root cells; a drift that is zero or beyond FP64's usual range
// is left out of the bins
static BinScale bin_scale(const LevelDev& root, double half_dt, int shift, int nb) {
    BinScale s;
    const double bin = std::ldexp(root.delta0, shift);
    int e = 0;
    std::frexp(root.box, &e);
    if (std::abs(e) > 800) e = 0;
    s.ex = e;
    s.cx = (float)(std::ldexp(1.0, e) / bin);
    int h = 0;
    const double f = std::frexp(half_dt, &h);
    const bool drift = half_dt != 0.0 && std::isfinite(half_dt) && std::abs(h) < 400 && std::abs(e) < 400;
    s.ev = drift ? e - h : 0;
    s.cv = drift ? (float)f * s.cx : 0.f;
    s.period = root.periodic ? (float)(root.box / bin) : 0.f;
    s.inv_period = root.periodic ? 1.f / s.period : 0.f;
    s.nb = nb;
    return s;
}

cudaError_t launch_order(const LevelDev& root, const Particles& P, double half_dt, int shift, int nb,
                         unsigned* count, unsigned* sums, unsigned* key, unsigned* rank, int* perm, cudaStream_t s) {
    if (P.n <= 0) return cudaSuccess;
    const int nbins = nb * nb * nb;
    const int nchunks = order_scan_chunks(nbins);
    if (nchunks > 1024) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(count, 0, (size_t)nbins * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)((P.n + 255) / 256);
    if ((e = launch_kernel(k_order_bins, blocks, 256, 0, s, P, bin_scale(root, half_dt, shift, nb), count, key,
                           rank)) != cudaSuccess ||
        (e = launch_kernel(k_order_scan_local, nchunks, 1024, 0, s, count, nbins, sums)) != cudaSuccess ||
        (e = launch_kernel(k_order_scan_sums, 1, 1024, 0, s, sums, nchunks)) != cudaSuccess)
        return e;
    return launch_kernel(k_order_scatter, blocks, 256, 0, s, P.n, key, rank, count, sums, perm);
}

}  // namespace apm
