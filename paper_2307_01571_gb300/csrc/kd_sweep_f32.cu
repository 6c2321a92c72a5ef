// Instantiates the fused sweep kernels for float spinors, one launch variant per object
// file: the build compiles this file once per KD_SWEEP_VARIANT so that the variants
// compile in parallel (kd_sweep_f32_forms.cu does the same for the forms beyond them).
#include "kd_sweep.cuh"

#ifndef KD_SWEEP_VARIANT
#define KD_SWEEP_VARIANT 0
#endif

namespace kd {
template <int V>
cudaError_t launch_sweep_f32_v(int axis, int shape, int logn, const SweepArgs& a, cudaStream_t s) {
    return launch_sweep<float, V>(axis, shape, logn, a, s);
}
template cudaError_t launch_sweep_f32_v<KD_SWEEP_VARIANT>(int, int, int, const SweepArgs&, cudaStream_t);

#if KD_SWEEP_VARIANT == 0
// the others are instantiated in their own objects
extern template cudaError_t launch_sweep_f32_v<1>(int, int, int, const SweepArgs&, cudaStream_t);
extern template cudaError_t launch_sweep_f32_v<2>(int, int, int, const SweepArgs&, cudaStream_t);
extern template cudaError_t launch_sweep_f32_v<3>(int, int, int, const SweepArgs&, cudaStream_t);
extern template cudaError_t launch_sweep_f32_v<kFormSmall>(int, int, int, const SweepArgs&, cudaStream_t);
extern template cudaError_t launch_sweep_f32_v<kFormLarge>(int, int, int, const SweepArgs&, cudaStream_t);
extern template cudaError_t launch_sweep_f32_v<kFormWide>(int, int, int, const SweepArgs&, cudaStream_t);
extern template cudaError_t launch_sweep_f32_v<kFormTall>(int, int, int, const SweepArgs&, cudaStream_t);
extern template cudaError_t launch_sweep_f32_v<kFormTallWide>(int, int, int, const SweepArgs&, cudaStream_t);

cudaError_t launch_sweep_f32(int form, int axis, int shape, int logn, const SweepArgs& a,
                             cudaStream_t s) {
    static_assert(kNumSweepVariants == 4 && kNumSweepForms == 9, "one case per compiled form");
    switch (form) {
        case 0: return launch_sweep_f32_v<0>(axis, shape, logn, a, s);
        case 1: return launch_sweep_f32_v<1>(axis, shape, logn, a, s);
        case 2: return launch_sweep_f32_v<2>(axis, shape, logn, a, s);
        case 3: return launch_sweep_f32_v<3>(axis, shape, logn, a, s);
        case kFormSmall: return launch_sweep_f32_v<kFormSmall>(axis, shape, logn, a, s);
        case kFormLarge: return launch_sweep_f32_v<kFormLarge>(axis, shape, logn, a, s);
        case kFormWide: return launch_sweep_f32_v<kFormWide>(axis, shape, logn, a, s);
        case kFormTall: return launch_sweep_f32_v<kFormTall>(axis, shape, logn, a, s);
        case kFormTallWide: return launch_sweep_f32_v<kFormTallWide>(axis, shape, logn, a, s);
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t build_twiddles_f32(int logn, int loge, void* out, int* entries, cudaStream_t s) {
    return build_twiddles<float>(logn, loge, out, entries, s);
}
#endif
}  // namespace kd
