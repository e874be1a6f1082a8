// k_fft_x.cu -- the x passes (xf, xi) of the batched FFT convolution and the
// shared-memory set-up of every pass kernel.
#include "fft_core.cuh"

namespace apm {

// the column passes' set-up (k_fft_col.cu, one per precision and pass)
cudaError_t fft_configure_yf_f32();
cudaError_t fft_configure_z_f32();
cudaError_t fft_configure_yi_f32();
cudaError_t fft_configure_yf_f64();
cudaError_t fft_configure_z_f64();
cudaError_t fft_configure_yi_f64();
cudaError_t fft_configure_zg_f32();
cudaError_t fft_configure_zg_f64();
// the passes with compile-time plans (k_fft_fast.cu, one unit per kernel,
// precision and group of lengths)
#define APM_FAST_DECL(m, p, g) \
    cudaError_t fast_launch##m##_##p##_##g(int L, const FftArgs& a, const int64_t* const* gmf, void* const* phis, \
                                           cudaStream_t s); \
    cudaError_t fast_configure##m##_##p##_##g(int L);
#define APM_FAST_F32(X, m) X(m, 0, 0) X(m, 0, 1) X(m, 0, 2) X(m, 0, 3)
#define APM_FAST_F64(X, m) X(m, 1, 1) X(m, 1, 2) X(m, 1, 3)
#define APM_FAST_UNITS(X) \
    APM_FAST_F32(X, 0) APM_FAST_F32(X, 1) APM_FAST_F32(X, 2) APM_FAST_F32(X, 3) APM_FAST_F32(X, 4) \
    APM_FAST_F32(X, 5) APM_FAST_F32(X, 6) APM_FAST_F32(X, 7) APM_FAST_F64(X, 0) APM_FAST_F64(X, 1) \
    APM_FAST_F64(X, 2) APM_FAST_F64(X, 3) APM_FAST_F64(X, 4) APM_FAST_F64(X, 5)
APM_FAST_UNITS(APM_FAST_DECL)

cudaError_t launch_fft_fast(int kernel, bool f64, int L, const FftArgs& a, const int64_t* const* gmf,
                            void* const* phis, cudaStream_t s) {
    const int u = (kernel * 2 + (f64 ? 1 : 0)) * kFastGroups + fast_group(L, f64);
#define APM_FAST_CASE(m, p, g) \
    case (m * 2 + p) * kFastGroups + g: return fast_launch##m##_##p##_##g(L, a, gmf, phis, s);
    if (fast_length(L, f64)) switch (u) { APM_FAST_UNITS(APM_FAST_CASE) }
#undef APM_FAST_CASE
    return cudaErrorInvalidValue;
}
cudaError_t configure_fft_fast(int kernel, bool f64, int L) {
    const int u = (kernel * 2 + (f64 ? 1 : 0)) * kFastGroups + fast_group(L, f64);
#define APM_FAST_CASE(m, p, g) \
    case (m * 2 + p) * kFastGroups + g: return fast_configure##m##_##p##_##g(L);
    if (fast_length(L, f64)) switch (u) { APM_FAST_UNITS(APM_FAST_CASE) }
#undef APM_FAST_CASE
    return cudaErrorInvalidValue;
}

// Allows every runtime-planned pass kernel up to kFftSmemLimit of dynamic shared memory
// (above the 48 KB default).
cudaError_t fft_configure() {
    const void* fns[] = {(const void*)k_xf<float, 128>, (const void*)k_xf<float, 256>,
                         (const void*)k_xi<float, 128>, (const void*)k_xi<float, 256>,
                         (const void*)k_xf<double, 128>, (const void*)k_xf<double, 256>,
                         (const void*)k_xi<double, 128>, (const void*)k_xi<double, 256>};
    for (const void* f : fns) {
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmemLimit);
        if (e != cudaSuccess) return e;
    }
    cudaError_t (*cols[])() = {fft_configure_yf_f32, fft_configure_z_f32, fft_configure_yi_f32,
                               fft_configure_zg_f32, fft_configure_yf_f64, fft_configure_z_f64,
                               fft_configure_yi_f64, fft_configure_zg_f64};
    for (auto f : cols) {
        cudaError_t e = f();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The CTA size is a template parameter of the pass kernels (128 or 256 threads).
template <typename T>
cudaError_t launch_fft_xf(const FftArgs& a, const int64_t* const* gmf, cudaStream_t s) {
    if (a.n_chunks <= 0) return cudaSuccess;
    if (a.threads == 128)
        return launch_kernel(k_xf<T, 128>, a.n_chunks, 128, a.smem, s, a.g, a.chunks, gmf, (const C<T>*)a.tw,
                             (C<T>*)a.wsA, a.F, a.status, a.inject_wait);
    else
        return launch_kernel(k_xf<T, 256>, a.n_chunks, 256, a.smem, s, a.g, a.chunks, gmf, (const C<T>*)a.tw,
                             (C<T>*)a.wsA, a.F, a.status, a.inject_wait);
}

template <typename T>
cudaError_t launch_fft_xi(const FftArgs& a, void* const* phis, cudaStream_t s) {
    if (a.n_chunks <= 0) return cudaSuccess;
    if (a.threads == 128)
        return launch_kernel(k_xi<T, 128>, a.n_chunks, 128, a.smem, s, a.g, a.chunks, (const C<T>*)a.tw,
                             (const C<T>*)a.wsB, phis, a.comp);
    else
        return launch_kernel(k_xi<T, 256>, a.n_chunks, 256, a.smem, s, a.g, a.chunks, (const C<T>*)a.tw,
                             (const C<T>*)a.wsB, phis, a.comp);
}

template cudaError_t launch_fft_xf<float>(const FftArgs&, const int64_t* const*, cudaStream_t);
template cudaError_t launch_fft_xf<double>(const FftArgs&, const int64_t* const*, cudaStream_t);
template cudaError_t launch_fft_xi<float>(const FftArgs&, void* const*, cudaStream_t);
template cudaError_t launch_fft_xi<double>(const FftArgs&, void* const*, cudaStream_t);

}  // namespace apm
