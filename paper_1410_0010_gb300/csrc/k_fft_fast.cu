// k_fft_fast.cu -- launchers of the FFT passes with compile-time plans
// (fft_fast.cuh), one per length of APM_FAST_LENGTHS_g; compiled once per
// kernel (enum kFastYf.., internal header), precision and group of lengths with
// -DAPM_FAST_MODE=0..7 -DAPM_FAST_FP64=0|1 -DAPM_FAST_GROUP=0..3, so the
// instantiations build in parallel.
// some members of Kern are used by some of the kernels only
#pragma nv_diag_suppress 177
#include "fft_fast.cuh"

#if !defined(APM_FAST_MODE) || !defined(APM_FAST_FP64) || !defined(APM_FAST_GROUP)
#error "k_fft_fast.cu is compiled with -DAPM_FAST_MODE=0..7 -DAPM_FAST_FP64=0|1 -DAPM_FAST_GROUP=0..3"
#endif

#define APM_FAST_CAT4(a, b, c, d) a##b##_##c##_##d
#define APM_FAST_NAME(a, b, c, d) APM_FAST_CAT4(a, b, c, d)
#define APM_FAST_CATL(g) APM_FAST_LENGTHS_##g
#define APM_FAST_LIST(g) APM_FAST_CATL(g)

namespace apm {

namespace {
using FT = typename std::conditional<APM_FAST_FP64, double, float>::type;
constexpr bool kF64 = APM_FAST_FP64;
constexpr int kMode = APM_FAST_MODE;
constexpr bool kFused = kMode == kFastXy || kMode == kFastYx;
constexpr int kLines = fast_lines(kF64);

// The plan of radices A, B, Cc.  FP64 takes 75 in three stages: 15 x 5 has 40 first
// butterflies in a CTA, one warp and a quarter, and the pipe that bounds it takes as
// long for the quarter as for a warp (8 grids of L = 75: 627 -> 514 us).
template <int A, int B, int Cc>
using PlanOf = typename std::conditional<kF64 && A * B * Cc == 75, FastPlan<3, 5, 5>, FastPlan<A, B, Cc>>::type;

template <int A, int B, int Cc>
struct Kern {
    using P = PlanOf<A, B, Cc>;
    static constexpr int L = A * B * Cc;
    static constexpr bool row = kMode == kFastXf || kMode == kFastXi;
    // a fused plane kernel exists where the plane fits the shared-memory limit
    static constexpr bool ok = !kFused || fast_xy_smem(L) <= (size_t)kFftSmemLimit;
    static constexpr int NT = kFused ? fast_xy_threads(kMode, L) : fast_threads(P::R1, P::R2, P::R3, kLines);
    static constexpr size_t smem = kFused ? fast_xy_smem(L) : (row ? fast_row_smem(L, kF64) : fast_col_smem(L, kF64));
    static constexpr auto get() {
        if constexpr (kMode == kFastYf) return k_col_fast<P, 1, 0, kLines, NT, FT>;
        else if constexpr (kMode == kFastZ) return k_col_fast<P, 2, 1, kLines, NT, FT>;
        else if constexpr (kMode == kFastYi) return k_col_fast<P, 1, 2, kLines, NT, FT>;
        else if constexpr (kMode == kFastZg) return k_col_fast<P, 2, 3, kLines, NT, FT>;
        else if constexpr (kMode == kFastXf) return k_xf_fast<P, kLines, NT, FT>;
        else if constexpr (kMode == kFastXi) return k_xi_fast<P, kLines, NT, FT>;
        else if constexpr (kMode == kFastXy) return k_xy_fast<P, NT>;
        else return k_yx_fast<P, NT>;
    }
};

template <int L, int A, int B, int Cc>
cudaError_t launch_one(const FftArgs& a, const int64_t* const* gmf, void* const* phis, cudaStream_t s) {
    using K = Kern<A, B, Cc>;
    static_assert(K::L == L, "plan length");
    if constexpr (K::ok) {
        constexpr auto kern = K::get();
        const auto* tw = (const C<FT>*)a.tw;
        if constexpr (kMode == kFastXf)
            return launch_kernel(kern, a.n_chunks, K::NT, K::smem, s, a.g, a.chunks, gmf, tw, (C<FT>*)a.wsA, a.F);
        else if constexpr (kMode == kFastXy)
            return launch_kernel(kern, a.n_chunks, K::NT, K::smem, s, a.g, a.chunks, gmf, tw, (C<FT>*)a.wsB, a.F);
        else if constexpr (kMode == kFastXi)
            return launch_kernel(kern, a.n_chunks, K::NT, K::smem, s, a.g, a.chunks, tw, (const C<FT>*)a.wsB, phis,
                                 a.comp);
        else if constexpr (kMode == kFastYx)
            return launch_kernel(kern, a.n_chunks, K::NT, K::smem, s, a.g, a.chunks, tw, (const C<FT>*)a.wsA, phis,
                                 a.comp);
        else
            return launch_kernel(kern, a.n_chunks, K::NT, K::smem, s, a.g, a.chunks, tw, (const FT*)a.tab,
                                 (C<FT>*)a.wsA, (C<FT>*)a.wsB, a.comp);
    }
    return cudaErrorInvalidValue;
}

template <int L, int A, int B, int Cc>
cudaError_t configure_one() {
    using K = Kern<A, B, Cc>;
    if constexpr (K::ok)
        return cudaFuncSetAttribute(K::get(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::smem);
    return cudaErrorInvalidValue;
}
}  // namespace

cudaError_t APM_FAST_NAME(fast_launch, APM_FAST_MODE, APM_FAST_FP64, APM_FAST_GROUP)(
    int L, const FftArgs& a, const int64_t* const* gmf, void* const* phis, cudaStream_t s) {
    if (a.n_chunks <= 0) return cudaSuccess;
    switch (L) {
#define APM_FAST_CASE(LL, A, B, Cc) \
    case LL: return launch_one<LL, A, B, Cc>(a, gmf, phis, s);
        APM_FAST_LIST(APM_FAST_GROUP)(APM_FAST_CASE)
#undef APM_FAST_CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t APM_FAST_NAME(fast_configure, APM_FAST_MODE, APM_FAST_FP64, APM_FAST_GROUP)(int L) {
    switch (L) {
#define APM_FAST_CASE(LL, A, B, Cc) \
    case LL: return configure_one<LL, A, B, Cc>();
        APM_FAST_LIST(APM_FAST_GROUP)(APM_FAST_CASE)
#undef APM_FAST_CASE
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace apm
