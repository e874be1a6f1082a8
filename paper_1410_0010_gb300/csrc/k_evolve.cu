// k_evolve.cu -- one timestep of the particles given accelerations evaluated at
// the half-step drifted positions x + v dt/2 (the drift of Sec. 2 that the
// deposit and interpolation apply): v' = v + a dt, x' = x + ((v + v')/2) dt,
// the drift-kick-drift leapfrog used to evolve the tests of Sec. 3.1 and 3.5
// without subcycling.  Every FP64 operation is explicitly rounded in this
// order, so the update is bit-identical to a plain IEEE evaluation.
#include "apm_internal.cuh"

namespace apm {
namespace {

// What bounds this kernel is the FP64 pipe (2 lanes per clock and SM, measured;
// a conversion to FP64 counts like an operation) next to its 108 bytes a particle
// (144 with FP64 accelerations): 7 operations per axis took 185 us for 4.2 M
// particles, the 5 that are left 137; FP64 accelerations, 6 to 5, 162 and 137.
// An FP32 acceleration is widened by moving its bits, and the half in
// ((v + v') / 2) dt goes into dt: halving is exact on either factor, so the
// product is rounded the same way.  Warps with a particle outside the ordinary
// range convert (a zero, subnormal, infinite or NaN acceleration) or halve the sum
// itself (one small enough to lose a bit, or a dt without a half), by integer
// operations: with FP64 ones there the compiler issues those of both sides (FP64
// accelerations: 205 us).
__device__ __forceinline__ bool ordinary(double) { return true; }
__device__ __forceinline__ bool ordinary(float a) { return ((__float_as_uint(a) >> 23) & 0xffu) - 1u < 254u; }
__device__ __forceinline__ double widen(double a) { return a; }
__device__ __forceinline__ double widen(float a) {
    const unsigned b = __float_as_uint(a);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// s / 2, rounded to nearest even where a subnormal result loses a bit
__device__ __forceinline__ double halved_any(double s) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(s), sign = b & (1ULL << 63), m = b ^ sign;
    if (m >= 0x7ffULL << 52) return s;                                  // infinite, NaN
    if (m >= 2ULL << 52) return __longlong_as_double((long long)(b - (1ULL << 52)));
    return __longlong_as_double((long long)(((m + ((m >> 1) & 1)) >> 1) | sign));
}

template <typename T>
__global__ void __launch_bounds__(256) k_kick_drift(long long n, double* __restrict__ x, double* __restrict__ y,
                                                    double* __restrict__ z, double* __restrict__ vx,
                                                    double* __restrict__ vy, double* __restrict__ vz,
                                                    const T* __restrict__ acc, double dt) {
    const unsigned block = begin_kernel();
    const long long i = (long long)block * blockDim.x + threadIdx.x;
    const bool live = i < n;
    const long long p = live ? i : n - 1;   // a thread past the end redoes the last particle, unstored
    // all nine loads first (the arrays are distinct), then the updates
    const double v[3] = {vx[p], vy[p], vz[p]};
    const double q[3] = {x[p], y[p], z[p]};
    const T at[3] = {acc[p], acc[n + p], acc[2 * n + p]};
    double a[3], vn[3], s[3], qn[3];
    bool plain = ordinary(at[0]) && ordinary(at[1]) && ordinary(at[2]);
    if (__all_sync(0xffffffffu, plain)) {
#pragma unroll
        for (int j = 0; j < 3; ++j) a[j] = widen(at[j]);
    } else {
#pragma unroll
        for (int j = 0; j < 3; ++j) a[j] = (double)at[j];
    }
    const double half_dt = __longlong_as_double(__double_as_longlong(dt) - (1LL << 52));   // dt / 2
    const unsigned de = ((unsigned)__double2hiint(dt) >> 20) & 0x7ffu;
    plain = de >= 2u && de < 0x7ffu;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        vn[j] = __dadd_rn(v[j], __dmul_rn(a[j], dt));
        s[j] = __dadd_rn(v[j], vn[j]);
        plain = plain && ((unsigned)__double2hiint(s[j]) & 0x7fffffffu) >= (2u << 20);
    }
    plain = __all_sync(0xffffffffu, plain);
    if (!plain) {
#pragma unroll
        for (int j = 0; j < 3; ++j) s[j] = halved_any(s[j]);
    }
    const double f = plain ? half_dt : dt;
#pragma unroll
    for (int j = 0; j < 3; ++j) qn[j] = __dadd_rn(q[j], __dmul_rn(s[j], f));
    if (!live) return;
    x[p] = qn[0];
    y[p] = qn[1];
    z[p] = qn[2];
    vx[p] = vn[0];
    vy[p] = vn[1];
    vz[p] = vn[2];
}

}  // namespace

template <typename T>
cudaError_t launch_kick_drift(long long n, double* x, double* y, double* z, double* vx, double* vy, double* vz,
                              const void* acc, double dt, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    return launch_kernel(k_kick_drift<T>, blocks, 256, 0, s, n, x, y, z, vx, vy, vz,
                         reinterpret_cast<const T*>(acc), dt);
}

template cudaError_t launch_kick_drift<float>(long long, double*, double*, double*, double*, double*, double*,
                                              const void*, double, cudaStream_t);
template cudaError_t launch_kick_drift<double>(long long, double*, double*, double*, double*, double*, double*,
                                               const void*, double, cudaStream_t);

}  // namespace apm
