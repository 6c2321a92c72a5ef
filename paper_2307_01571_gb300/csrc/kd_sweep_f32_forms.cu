// The FP32 sweeps' forms beyond the launch variants (sweep_form in kd_internal.h: small,
// tall, large and the wide ones), compiled once per KD_SWEEP_FORM for the axis lengths that use them.
#include "kd_sweep.cuh"

namespace kd {
template <int V>
cudaError_t launch_sweep_f32_v(int axis, int shape, int logn, const SweepArgs& a, cudaStream_t s) {
    return launch_sweep<float, V>(axis, shape, logn, a, s);
}
template cudaError_t launch_sweep_f32_v<KD_SWEEP_FORM>(int, int, int, const SweepArgs&, cudaStream_t);
}  // namespace kd
