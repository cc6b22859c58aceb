// Mixed-precision trace kernels (OSIRIS_MIXED), Kerr and the q-metric: the
// lane state machine of the DF64 kernels (trace_df_body.cuh) with the six
// evaluations of Hamilton's equations of every attempt in FP32 (rhs_f32.cuh)
// and a stepper that sums their derivatives in FP32 (step_mixed.cuh). The
// state and the stage inputs keep df64 precision (FP32 with compensated
// sums), so adding a small increment to the state loses nothing; the
// derivatives carry FP32 rounding, ~1e-7 of |k|, and the sums over stages
// (increments, error estimate) add roundings of the same relative size. No
// step of the integration runs on the FP64 pipe: FP64 only sets up each ray,
// keeps the step-length bracket of surface location and forms the outputs.
//
// Tolerance range. The embedded error estimate h sum_s (b_s - b*_s)(k_s - k_1)
// then carries a noise of ~1e-8 h |k| ~ 1e-8 (h/tau) |y| (tau: time scale of
// the solution), against the local error tol (1 + |y|) that the controller
// compares it with. At tol 1e-8 the accepted steps have h/tau ~ 0.03 and the
// noise is a few percent of the estimate; at 1e-10 it is as large as the
// estimate and the controller would shrink the steps to chase it. MIXED is
// meant for tolerances of 1e-8 and looser; DF64 covers the tighter ones.
//
// |H|. The FP32 evaluations' own 2H carries the rounding of its largest terms
// (P^2 / Delta grows without bound towards the horizon), so it does not track
// the constraint; a ray's |H| output is that of its end point, evaluated in
// double-float (rhs_df) as in the DF64 kernels.
//
// Surface location. A trial step's end point carries the FP32 rounding of its
// stage derivatives, ~1e-7 h |k|, so the step-length bracket is resolved to a
// relative width of 2e-7, not to the DF64 kernels' 4e-16.
#include <cuda_runtime.h>

#include "rhs_f32.cuh"
#include "trace_df_body.cuh"

namespace osiris_impl {

// Registers. Large launches are bound by issue slots and gain from warps that
// hide the dependent FP32 chains: 80 registers (six blocks of 128 threads per
// SM) for Kerr, 128 (four) for the q-metric. Measured at tol 1e-8 on the
// 12 x 1024^2 Kerr set (Mrays/s, Cash-Karp, refill at 32 idle lanes): 96
// registers 160.9, 80: 162.3, 72: 154.7, 64: 153.0; on six 500^2 q-metric
// renders in one launch (ms) 56 registers 13.8, 80: 14.6, 104: 14.5, 128: 12.7,
// no cap 13.5, on a 1024^2 render 9.45 / 9.47 / 10.1 / 9.17 / 9.9. Small
// launches last as long as their longest chains: no cap (145-160 registers,
// three blocks per SM), nothing spilled. 80 / no cap, in ms, for Kerr:
//   render     32^2  0.80 / 0.62    256^2  1.13 / 0.99    512^2  2.37 / 2.29
//             800^2  4.32 / 4.58
//   disk      200^2  1.08 / 0.89    500^2  1.85 / 1.82    900^2  4.51 / 4.91
//   six renders in one launch  100^2  1.33 / 1.12    200^2  2.51 / 2.52    400^2  7.2 / 7.6
//   Dormand-Prince render      200^2  1.13 / 0.89    400^2  1.76 / 1.66    800^2  4.46 / 4.81
// and 128 / no cap for the q-metric: 100^2 0.89 / 0.82, 300^2 1.68 / 1.60, 600^2
// 3.69 / 3.94, six 200^2 renders 2.89 / 2.93. The lines lie at 5 and 2.5 times
// 256 lanes on each of 152 SMs.
constexpr int64_t kLargeLaunchKerr = 5 * 152 * 256;
constexpr int64_t kLargeLaunchQ = 5 * 152 * 256 / 2;

template <bool kTiny>
struct KerrMixed {
  using Ray = RayF32;
  static constexpr int kMaxRegs = 80;
  static constexpr bool kFusedR2 = false;
  static constexpr bool kTrackH = false;
  static constexpr bool kF32Stages = true;
  static constexpr double kLocateRel = 2e-7;
  static __device__ __forceinline__ Ray ray(const RayK& K) {
    Ray k;
    k.a = (float)K.a;
    k.a2 = (float)K.a2;
    k.aE = (float)K.aE;
    k.aL = (float)K.aL;
    k.E = (float)K.E;
    k.L = (float)K.L;
    k.twoE = (float)(2.0 * K.E);
    const double sq = sqrt(fmax(0.0, 1.0 - K.a2));
    k.rp = df_from_double(1.0 + sq);
    k.rm = (float)(1.0 - sq);
    k.twoH0 = 0.0f;
    return k;
  }
  static __device__ __forceinline__ void rhs_f(const Ray& K, const PointF32& x, float& dr,
                                               float& dth, float& dph, float& dpr, float& dpth,
                                               float& twoH) {
    rhs_f32<kTiny>(K, x, dr, dth, dph, dpr, dpth, twoH);
  }
  // 2 (H - H0) at the end point with the double-float equations of DF64.
  static __device__ __forceinline__ float end_twoH(const Ray& KD, const RayK& K,
                                                   const StateDF& y) {
    RayDF k = to_df(K);
    k.twoH0 = KD.twoH0;
    df dr, dth, dph, dpr, dpth;
    float twoH;
    rhs_df(k, y.r, y.th, y.pr, y.pth, dr, dth, dph, dpr, dpth, twoH);
    return twoH;
  }
};

// The q-metric (Appendix A) with the same stepper; its end-point |H| from
// the double-float q-metric equations (rhs_q_df).
template <bool kTiny>
struct QMetricMixed {
  using Ray = RayQF32;
  static constexpr int kMaxRegs = 128;
  static constexpr bool kFusedR2 = false;
  static constexpr bool kTrackH = false;
  static constexpr bool kF32Stages = true;
  static constexpr double kLocateRel = 2e-7;
  static __device__ __forceinline__ Ray ray(const RayK& K) {
    Ray k;
    k.E = (float)K.E;
    k.L = (float)K.L;
    k.q = (float)K.q;
    k.kap = (float)K.kap;
    k.nq1 = (float)(-(1.0 + K.q));
    k.E2 = (float)(K.E * K.E);
    k.twoH0 = 0.0f;
    return k;
  }
  static __device__ __forceinline__ void rhs_f(const Ray& K, const PointF32& x, float& dr,
                                               float& dth, float& dph, float& dpr, float& dpth,
                                               float& twoH) {
    rhs_q_f32<kTiny>(K, x, dr, dth, dph, dpr, dpth, twoH);
  }
  static __device__ __forceinline__ float end_twoH(const Ray& KD, const RayK& K,
                                                   const StateDF& y) {
    RayQDF k = to_qdf(K);
    k.twoH0 = KD.twoH0;
    df dr, dth, dph, dpr, dpth;
    float twoH;
    rhs_q_df(k, y.r, y.th, y.pr, y.pth, dr, dth, dph, dpr, dpth, twoH);
    return twoH;
  }
};

template <class Met, int INTEG, bool kLarge>
__global__ void __maxnreg__(kLarge ? Met::kMaxRegs : 255)
    trace_mixed_plain(const __grid_constant__ KernelArgs A) {
  trace_body_df<Met, Kernel::kPlain, INTEG>(A);
}

template <class Met, int INTEG, bool kLarge>
__global__ void __maxnreg__(kLarge ? Met::kMaxRegs : 255)
    trace_mixed_persistent(const __grid_constant__ KernelArgs A) {
  trace_body_df<Met, Kernel::kPersistent, INTEG>(A);
}

template <class Met, int INTEG, bool kLarge>
static const void* mixed_kernel(Kernel kind) {
  return kind == Kernel::kPersistent ? (const void*)trace_mixed_persistent<Met, INTEG, kLarge>
                                     : (const void*)trace_mixed_plain<Met, INTEG, kLarge>;
}

template <template <bool> class Met, int INTEG>
static const void* mixed_kernel(Kernel kind, int64_t rays, int64_t line) {
  if (kind == Kernel::kTinyRound)
    return (const void*)trace_mixed_persistent<Met<true>, INTEG, true>;
  return rays >= line ? mixed_kernel<Met<false>, INTEG, true>(kind)
                      : mixed_kernel<Met<false>, INTEG, false>(kind);
}

template <template <bool> class Met>
static const void* mixed_kernel(Kernel kind, int integrator, int64_t rays, int64_t line) {
  return integrator == OSIRIS_RKDP45 ? mixed_kernel<Met, OSIRIS_RKDP45>(kind, rays, line)
                                     : mixed_kernel<Met, OSIRIS_RKCK45>(kind, rays, line);
}

const void* trace_kernel_mixed(Kernel kind, int integrator, int spacetime, int64_t rays) {
  return spacetime == OSIRIS_SPACETIME_QMETRIC
             ? mixed_kernel<QMetricMixed>(kind, integrator, rays, kLargeLaunchQ)
             : mixed_kernel<KerrMixed>(kind, integrator, rays, kLargeLaunchKerr);
}

}  // namespace osiris_impl
