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

// Registers. Small launches last as long as their longest chains: no cap
// (three blocks of 128 threads per SM), nothing spilled. Large launches are
// bound by issue slots and gain from warps that hide the dependent FP32 chains:
// 96 registers (five blocks) for Kerr, 128 (four) for the q-metric (earlier
// sweeps: Kerr 72 and 64 slower than 80, q-metric 56 and 80 slower than 128).
// Kerr, 80 / 96 / no cap, ms at tol 1e-8:
//   render   360^2  1.35 / 1.37 / 1.21    512^2  2.10 / 2.02 / 1.96    640^2  3.01 / 2.93 / 2.84
//            800^2  3.92 / 3.91 / 4.01   1024^2  6.19 / 6.17 / 6.40   2048^2 22.83 / 22.78 / 23.44
//   disk     400^2  1.21 / 1.17 / 1.14    600^2  2.11 / 2.10 / 2.17   2048^2 19.46 / 19.54 / 20.85
//   six renders in one launch  200^2  2.20 / 2.17 / 2.13   400^2  6.59 / 6.52 / 6.62
//                              800^2 23.57 / 23.13 / 23.77
//   particles  100,000  0.366 / 0.349 / 0.326    400,000  0.960 / 0.951 / 0.977
//   Dormand-Prince render      400^2  1.56 / 1.55 / 1.45   1024^2 6.50 / 6.53 / 6.69
// q-metric, 128 / 104 / no cap:
//   render   300^2  1.46 / 1.51 / 1.27    400^2  1.91 / 2.01 / 1.79    512^2  2.64 / 2.86 / 2.67
//            600^2  3.29 / 3.62 / 3.34   1024^2  8.17 / 8.91 / 8.46
//   six renders in one launch  200^2  2.55 / 2.68 / 2.52   500^2 11.5 / 12.4 / 11.9
// The lines lie at 8 and 5 times 256 lanes on each of 152 SMs.
constexpr int64_t kLargeLaunchKerr = 8 * 152 * 256;
constexpr int64_t kLargeLaunchQ = 5 * 152 * 256;

struct KerrMixed {
  using Ray = RayF32;
  static constexpr int kMaxRegs = 96;
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
    rhs_f32(K, x, dr, dth, dph, dpr, dpth, twoH);
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
    rhs_q_f32(K, x, dr, dth, dph, dpr, dpth, twoH);
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

template <class Met, int INTEG>
static const void* mixed_kernel(Kernel kind, int64_t rays, int64_t line) {
  return rays >= line ? mixed_kernel<Met, INTEG, true>(kind)
                      : mixed_kernel<Met, INTEG, false>(kind);
}

template <class Met>
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
