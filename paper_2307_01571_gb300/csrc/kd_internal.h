// kd_internal.h -- declarations shared by the host API (kd_api.cu) and the sweep kernels
// (kd_sweep_f32.cu, kd_sweep_f64.cu).  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace kd {

// Lets kernel k take `bytes` of dynamic shared memory on the current device.  The limit belongs
// to one device's copy of the kernel: `done` holds one bit per device that accepted it (devices
// beyond the 64th are asked every time).
template <typename K> cudaError_t allow_smem(K k, int bytes, std::atomic<uint64_t>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
    if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

// Internal spinor layout: two pair planes [pair][ny][nx][2] complex.  In 2D with
// A = (A_x, A_y) and p = (p_x, p_y) both alpha.A and alpha.p + beta couple only
// psi1 <-> psi4 and psi2 <-> psi3, so the problem splits exactly into pair 0 = (psi1, psi4)
// and pair 1 = (psi2, psi3); internal slot s = 2 pair + index within the pair.  Pair 1's
// 2x2 generators are pair 0's with the y component negated.
__host__ __device__ constexpr int perm_to_dirac(int s) {  // internal slot -> Dirac component
    return s == 0 ? 0 : (s == 1 ? 3 : (s == 2 ? 1 : 2));
}

enum SweepAxis { AXIS_X = 0, AXIS_Y = 1 };
// FFT presence: FFT1 runs before the pointwise op, FFT2 after it.  On the x axis FFT1
// is inverse and FFT2 forward; on the y axis FFT1 is forward and FFT2 inverse.
enum SweepShape { SHAPE_F2 = 1, SHAPE_F1 = 2, SHAPE_F1F2 = 3 };
enum SweepOp { OP_NONE = 0, OP_POTENTIAL = 1, OP_KINETIC = 2 };

// Per-step scalars, FP64, written once per kd_step by a small kernel.
struct StepScalars {
    double t;      // time of the step boundary
    double s;      // a0 f(t) sin(omega t + phase0): common factor of the standing wave
    double ybase;  // y of row 0: y_min + box_vy t (co-moving box)
    float s_f;     // the same two, rounded once for the FP32 sweeps
    float ybase_f;
};

// Device clock: absolute step index of the state and the index at the start of the
// current kd_step call.  Kernels index StepScalars with (step - base) + n_local.
struct Clock {
    long long step;
    long long base;
};

struct SweepArgs {
    const void* in;
    void* out;
    const void* tw;       // stage-major twiddle table (build_twiddles_*): double2 (FP64)
                          // or float4 (c_hi, s_hi, c_lo, s_lo) (FP32)
    int nx, ny;
    int op;
    // potential (x sweep)
    const Clock* clock;
    const StepScalars* steps;
    int n_local;
    int kind, longitudinal;
    double kappa;         // tau m c^2 / hbar for this sweep (tau = dt or dt/2)
    double eps4;          // 4 epsilon (longitudinal amplitude factor)
    double y_min, dy;
    // FP32 copies of the scalars, rounded once on the host, so that the FP32 sweeps do
    // no FP64 arithmetic (the FP64 pipe is 1/64 of FP32 on GB300)
    float kappa_f, eps4_f, dy_f, mc_f, invP_f;
    double invP;          // 1 / (nx ny), exact
    const void* xtab;     // [2][nx][4] per-x field table, precision of the sweep:
                          // (Theta0, x/(x_R w^2), w0/w, 1/w^2) then (1/w, cos zeta, sin zeta, cos k x)
    // kinetic (y sweep)
    const void* ktab;     // [ny][nx] (C/P, c S/P) pairs
    const void* kxtab;    // [nx] pi_x
    const void* kytab;    // [ny] (pi_y, cos, sin of the frame phase, pad)
    double mc;            // m c
    // precision form (tensor-core sweeps of 1024-point axes, kd_tc.cu)
    const void* tc_b;     // 32-point DFT matrices (inverse hi, lo, forward hi, lo), FP16,
                          // times 2^10, in the kernel's shared-memory image (32 KiB)
    const void* tc_tw;    // [1024] float2 (cos, sin) of 2 pi m / 1024
    const float* tc_scale;  // [axis][2] power-of-two operand scales, set per kd_step
    const void* dwconst;  // double-word form: constant tables of exp and sin/cos (DWConst)
    int* status;          // error word of the simulation (KD_STATUS_* bits)
    int tc_fault;         // test hook (kd_inject_fault): the tensor-core sweep issues no
                          // matrix products, so that its bounded waits run out
};

// bits of the device status word
constexpr int KD_STATUS_NONFINITE = 1, KD_STATUS_DRIFT = 2, KD_STATUS_TC_TIMEOUT = 16;

// Launch variants of the FP32 sweeps, timed per grid by the autotuner (kd_autotune);
// variant 0 is the default.  The table is what 2 and 3 always run and 0 and 1 run where
// sweep_form_of (below) has nothing better for the grid's size.  A variant fixes the radix schedule (loge = log2 of the
// elements a thread owns: radix-8 or radix-4 Stockham stages), the threads per CTA (a
// target: at least one whole line), the minimum column-tile width of the y sweep, the
// spinor components per CTA (2: one 2x2 pair per CTA, the two pairs' CTAs side by side;
// 4: both pairs, sharing the field or table loads) and the resident warps per SM the
// register budget is built for.  Variants that differ only in threads or tile width do
// the same arithmetic per line (bitwise identical results); a different radix schedule,
// or components per CTA (the compiler may fuse the pointwise ops' multiply-adds
// differently), rounds differently.  share (x axis, nc 2): one CTA holds both pairs of its
// lines, the pairs' threads owning the same points; each thread evaluates the standing
// wave for half of its points and the two halves trade the potential factors through
// shared memory (the field costs as much as both pairs' arithmetic of the potential step).
// FP64 sweeps have the one variant 0.
struct SweepVariant {
    int loge, threads, minb, nc, resident_warps, share;
};
constexpr int kNumSweepVariants = 4;
__host__ __device__ constexpr SweepVariant sweep_variant(int axis, int v) {
    return axis == AXIS_X
        ? (v == 1 ? SweepVariant{3, 256, 1, 2, 24, 1}
         : v == 2 ? SweepVariant{2, 128, 1, 2, 32, 0}
         : v == 3 ? SweepVariant{3, 128, 1, 4, 16, 0}
                  : SweepVariant{3, 128, 1, 2, 28, 0})
        : (v == 1 ? SweepVariant{3, 512, 8, 4, 16, 0}
         : v == 2 ? SweepVariant{2, 256, 4, 4, 24, 0}
         : v == 3 ? SweepVariant{3, 256, 4, 2, 28, 0}
                  : SweepVariant{3, 256, 4, 4, 16, 0});
}
// spinor components per thread of the FP32 sweeps
__host__ __device__ constexpr int sweep_nc(int axis, int v);

// The compiled forms of the FP32 sweeps: 0 ... 3 the variants as in the table, and those that
// the default (variants 0 and 1) becomes by the grid's size, sweep_form_of below.
//   small: radix-4 stages, one or two rows / two columns per CTA.  A small grid is bound by
//     the latency of one CTA and by idle SMs: 128 columns of 128 points in tiles of eight
//     columns and both pairs were 16 CTAs on 152 SMs.
//   tall (columns): radix-8 stages, one column per CTA, for at most 32 columns of 1024 and 2048
//     points, where three stages instead of five or six outweigh the 16-byte rows of the tile
//     (us a step, small : tall: 16x1024 9.91 : 9.46, 32x1024 10.00 : 9.75, 32x2048 13.85 :
//     13.59; but 64x1024 11.1 : 14.8).
//   large (columns): radix-16 stages, sixteen elements a thread.  A grid of many rounds is
//     bound by the shared-memory exchanges and twiddle loads together with the FP32 pipe;
//     radix-16 stages take two thirds of the former, and many rounds make up for the fewer
//     warps.  (Rows gain more from both pairs per thread, which evaluates the field once.)
//   wide, tall wide: what members of a batch that fills the SMs run in the place of small and of
//     the long columns' forms: both pairs per thread, rows in CTAs of 256 threads, columns in
//     tiles of 256 threads (two columns at 512 points, where four would take 512).
// All radix-4 rows round alike, and so do small and wide columns, and tall wide ones with tall
// and, from 1024 points, variant 3: their pointwise steps have every fusion written out, so that
// components per thread do not change a bit.
constexpr int kFormSmall = 4, kFormLarge = 5, kFormWide = 6, kFormTall = 7, kFormTallWide = 8, kNumSweepForms = 9;
__host__ __device__ constexpr SweepVariant sweep_form(int axis, int form) {
    if (form < kNumSweepVariants) return sweep_variant(axis, form);
    if (form == kFormWide) return axis == AXIS_X ? SweepVariant{2, 256, 1, 4, 24, 0} : SweepVariant{2, 256, 2, 4, 24, 0};
    if (form == kFormTall) return SweepVariant{3, 64, 1, 2, 28, 0};
    if (form == kFormTallWide) return SweepVariant{3, 256, 4, 4, 16, 0};
    if (axis == AXIS_X) return SweepVariant{2, 64, 1, 2, 32, 0};
    return form == kFormSmall ? SweepVariant{2, 64, 2, 2, 32, 0} : SweepVariant{4, 256, 2, 2, 16, 0};
}
// axes and lengths a form is compiled for: those at which sweep_form_of gives it on some grid
// (axes end at 4096 points)
__host__ __device__ constexpr bool sweep_form_holds(int axis, int form, int logn) {
    return form <= 1               ? (axis == AXIS_X ? logn >= 7 : logn >= 6 && logn <= 9)
           : form == kFormSmall    ? logn <= (axis == AXIS_X ? 11 : 10)
           : form == kFormWide     ? logn <= (axis == AXIS_X ? 11 : 9)
           : form == kFormTall     ? axis == AXIS_Y && (logn == 10 || logn == 11)
           : form == kFormTallWide ? axis == AXIS_Y && logn >= 10
           : form == kFormLarge    ? axis == AXIS_Y && logn >= 10
                                   : true;
}
// The form that variant v runs on `lines` lines of 2^logn points.  The lines lie where the
// times of whole runs cross (GB300, us per step, both sweeps; a sweep timed alone can mislead:
// variant 1's 512-thread rows are the fastest at 2048x128 alone, 10.3 against 10.9 us, but leave
// no room for the next sweep to start under, 21.8 against 19.5 a step).  Variant 0 : chosen:
//   x small up to 2^16 points, for short rows up to 2^18 (with the chosen columns: 64x64 10.4 :
//     5.3, 128x128 11.7 : 6.0, 256x256 13.4 : 8.6, 256x1024 21.1 : 17.3, 128x2048 22.0 : 18.8);
//   x 512 and 1024 points at 2^17: variant 1, the field shared in a CTA (512x256 15.0 : 11.4,
//     1024x128 15.3 : 11.5); at 2^18 and beyond variant 0 (512x512 18.7, small 22.2);
//   x 2048 and 4096 points: both pairs per thread (variant 3) from 2^18 and 2^19 points on
//     (2048x128 23.8 : 19.5, 2048x256 30.9 : 27.7; with large columns 2048x1024 118.2 : 118.0,
//     2048x2048 267 : 252, 4096x2048 562 : 522; radix-16 rows 129, 265, 529); 4096x64 is too
//     few rows for it (a sweep 11.1 : 16.7);
//   x 2048 points at 2^17: variant 0 (13.1 with small rows, 11.9);
//   y small up to 2^16 points (2^15 at 512, tall for few columns of 1024 and more), radix-4
//     tiles of both pairs (wide) at 2^17 up to 256 points; one pair per CTA (variant 3) for few
//     long columns (128x512 12.1 : 10.3, 256x512 15.3 : 12.3, 128x1024 20.9 : 15.2, 64x2048
//     23.5 : 16.3, 256x1024 24.1 : 17.3 with small rows); large beyond (1024x1024 56.5 : 55.0,
//     2048x1024 125.5 : 118.2, 4096x2048 589 : 562).
// crowded: other simulations run beside this one and fill the SMs (a batch).  The narrow tiles
// that spread one small grid over the SMs then only cost: the field, the twiddles and the index
// work of each pair of components, and memory transactions.  The wide forms take their place,
// with the same arithmetic, so that a member still equals itself run alone, bit for bit (which
// rules the radix-8 shapes out where a grid alone runs radix-4 stages).  G point-steps/s of a
// batch, its members' forms when alone (columns: variant 2's tiles) : radix-8 shapes of the
// table's variant 0 : here:
//   256 of 256x128 20.9 : 22.7 : 22.8, 256 of 128x128 17.3 : 18.0 : 18.6, 64 of 256x256 20.4 :
//   22.1 : 21.9, 64 of 128x512 19.8 : 21.0 : 21.7, 64 of 1024x64 20.4 : 23.0 : 24.1, 32 of
//   32x2048 14.3 : 19.7 : 20.3, 32 of 128x1024 17.7 : 19.3 : 19.6, 64 mixed 20.1 : 19.4 : 20.6;
//   radix-4 stages of 512 points and more, and 256-point columns at 2^17 points, stay behind:
//   64 of 64x512 18.6 : 24.3 : 21.4, 64 of 64x1024 16.6 : 19.3 : 16.7, 32 of 512x256 22.4 :
//   23.3 : 22.5 (alone these grids take 7.5, 11.1 and 11.6 us a step; variant 0's shapes 12.9,
//   20.6 and 15.0).
inline int sweep_form_of(int axis, int v, int logn, int lines, bool crowded) {
    if (v > 1) return v;
    int logp = logn;   // log2 of the points (both counts are powers of two)
    while ((lines >> (logp - logn)) > 1) ++logp;
    if (axis == AXIS_X) {
        const int small = crowded ? kFormWide : kFormSmall;
        if (logn <= 8) return logp <= 18 ? small : v;
        if (logn <= 10) return logp <= 16 ? small : (logp == 17 ? 1 : v);
        if (logn == 11) return logp <= 16 ? small : (logp == 17 ? v : 3);
        return logp <= 18 ? v : 3;
    }
    if (logn <= 9) {
        if (logp <= (logn == 9 ? 15 : 16)) return crowded ? kFormWide : kFormSmall;
        return logp <= 17 ? (logn == 9 ? 3 : kFormWide) : v;
    }
    if (logp > 18) return kFormLarge;
    if (lines == 64 && logn == 10) return kFormSmall;
    return crowded ? kFormTallWide : (logp <= 16 && logn <= 11 ? kFormTall : 3);
}

__host__ __device__ constexpr int sweep_nc(int axis, int v) { return sweep_form(axis, v).nc; }
// log2 of the elements per thread (the radix of the Stockham stages): FP32, FP64
__host__ __device__ constexpr int sweep_loge(int axis, int logn, int v) {
    const int lmax = sweep_form(axis, v).loge;
    return logn < lmax ? logn : lmax;
}
// radix-4 stages up to 1024 points, radix-8 above, so that a line's threads stay within 256
// (512 at 4096) and two lines fit on an SM
__host__ __device__ constexpr int sweep_loge_f64(int logn) { return logn < 2 ? logn : (logn <= 10 ? 2 : 3); }

// log2 of the elements per thread of the double-word form: radix-4 stages (four
// double-word complex values per component keep the register use within two CTAs per SM)
// up to 1024-point lines, radix-8 above (a line's threads stay within 256)
__host__ __device__ constexpr int sweep_loge_dw(int logn) { return logn < 2 ? logn : (logn <= 10 ? 2 : 3); }

// Launches one sweep; returns cudaSuccess or the launch error.  logn in [2, 12], form in
// [0, kNumSweepForms) and compiled for logn.
template <int V>
cudaError_t launch_sweep_f32_v(int axis, int shape, int logn, const SweepArgs& a, cudaStream_t s);
cudaError_t launch_sweep_f32(int form, int axis, int shape, int logn, const SweepArgs& a,
                             cudaStream_t s);
cudaError_t launch_sweep_f64(int axis, int shape, int logn, const SweepArgs& a, cudaStream_t s);
// Double-word form (KD_DW): the FP64 form's launch shapes with every real a float pair.
cudaError_t launch_sweep_dw(int axis, int shape, int logn, const SweepArgs& a, cudaStream_t s);
// Precision form: whether an axis of 2^logn points has the tensor-core sweep, and its
// launch (full sweeps only; persistent, at most two CTAs per SM).
bool tc_supported(int logn);
cudaError_t launch_tc_sweep(int axis, const SweepArgs& a, cudaStream_t s);
// Fills the stage-major twiddle table of an N = 2^logn sweep whose threads own 2^loge
// elements (at most 2N entries of 16 B) and returns the number of entries.
cudaError_t build_twiddles_f32(int logn, int loge, void* out, int* entries, cudaStream_t s);
cudaError_t build_twiddles_f64(int logn, int loge, void* out, int* entries, cudaStream_t s);
cudaError_t build_twiddles_dw(int logn, int loge, void* out, int* entries, cudaStream_t s);

}  // namespace kd
