// Double-float trace kernels. Every Cash-Karp attempt of the integration runs
// in df64 arithmetic (pairs of FP32, 48-bit significand) on the FP32 pipe,
// which on GB300 is ~70x the FP64 pipe: the six evaluations of Hamilton's
// equations, the stage sums, the increment, the error estimate, the error
// test, the stopping-surface tests and the end-point |H|. The state between
// steps is a df64 vector too. FP64 is used only once per ray (initial data,
// the terminal state and the observables) and for the step-length bracket of
// surface location.
//
// Stage sums. With d_j = k_j - k_1 (j >= 2), the Cash-Karp combinations are
//   stage input  y_i = y + c_i h k_1 + h sum_j a_ij d_j      (sum_j a_ij = c_i)
//   increment        = h k_1 + h sum_i b_i d_i                (sum_i b_i = 1)
//   error estimate   = h sum_i (b_i - b*_i) d_i               (sum = 0)
// The increment is formed in df64 with df64 weights. The error estimate
// cancels to O(h^5), but every d_i is exact to df64 precision, so the leading
// words summed in FP32 keep its relative error near 2^-24 (h/T)^-3 / 30 (T:
// time scale of the solution), a fraction of a percent at tol 1e-10 (the
// derivation is at rk_step_df). In a stage input the part h sum_j a_ij d_j
// is O(h/T) smaller than the stage's step and reaches the result only
// through one more factor h/T, so it is summed in FP32 too.
//
// The six stages run as a loop with one copy of the evaluation of Hamilton's
// equations (six inlined df64 copies overflow the instruction cache), and
// every stage sum is kept in registers.
//
// The evaluations (Kerr and q-metric) are in rhs_df.cuh, the attempt and its
// tableaus in step_df.cuh, the lane state machine in trace_df_body.cuh; this
// file holds the double-float metric policies and the launchers.
#include "trace_df_body.cuh"

namespace osiris_impl {

// Metric policies of the double-float kernels: the ray constants, the
// evaluation, and the register cap.
//
// Two variants, chosen by the launch's rays. Small launches have one or two
// warps per SM sub-partition and last as long as their longest chains: no cap
// (203-234 registers, two blocks of 128 threads per SM), nothing spilled.
// Large launches: 128 registers, so that four blocks are resident per SM: the
// double-float dependency chains gain more from the extra warps than they lose
// to the spilled values, which stay in L1 as long as no shared memory is
// reserved. 128 registers / 168 (three blocks) / no cap, ms:
//   Kerr render  100^2  4.7 / - / 3.0      360^2   9.7 / 9.2 / 8.3    512^2  15.4 / 15.1 / 14.0
//                640^2 21.9 / 21.9 / 20.6  800^2  31.0 / 30.9 / 30.7  2048^2 184.6 / 185.9 / 187.4
//   disk         400^2  8.5 / 8.1 / 8.0    600^2  15.5 / 15.4 / 15.2  2048^2 153.7 / 155.3 / 158.2
//   six renders  200^2 15.9 / 15.9 / 14.9  400^2  51.2 / 50.4 / 50.8  800^2 189.0 / 189.1 / 194.0
//   particles    100,000  2.33 / 1.99 / 1.83      400,000  5.74 / 5.68 / 5.88
//   Dormand-Prince render     400^2 12.4 / 13.2 / 10.9   1024^2 56.3 / 57.9 / 56.7
//   q-metric     300^2 15.8 / 15.5 / 13.5  512^2  27.3 / 28.3 / 27.0  600^2  34.3 / 35.6 / 34.5
//               1024^2 82.4 / 87.2 / 88.0  six 200^2 27.1 / 27.6 / 27.0
// The lines lie at 10 (Kerr) and 8 (q-metric) times the lanes that the uncapped
// kernels keep in flight (256 on each of 152 SMs), where the first kind of
// launch gets no slower by the cap (Kerr particles, q-metric renders).
constexpr int64_t kLargeLaunchKerr = 10 * 152 * 256;
constexpr int64_t kLargeLaunchQ = 8 * 152 * 256;
constexpr int kLargeRegs = 128;

struct KerrDF {
  using Ray = RayDF;
  static constexpr int kMaxRegs = kLargeRegs;
  static constexpr bool kFusedR2 = true;
  static __device__ __forceinline__ Ray ray(const RayK& K) { return to_df(K); }
  static __device__ __forceinline__ void rhs(const Ray& K, df r, df th, df pr, df pth, df& dr,
                                             df& dth, df& dph, df& dpr, df& dpth,
                                             float& twoH) {
    rhs_df(K, r, th, pr, pth, dr, dth, dph, dpr, dpth, twoH);
  }
  static constexpr bool kTrackH = true;
  static constexpr bool kF32Stages = false;
  static constexpr double kLocateRel = 4e-16;
  static __device__ __forceinline__ float end_twoH(const Ray& K, const RayK&, const StateDF& y) {
    df dr, dth, dph, dpr, dpth;
    float twoH;
    rhs(K, y.r, y.th, y.pr, y.pth, dr, dth, dph, dpr, dpth, twoH);
    return twoH;
  }
};

struct QMetricDF {
  using Ray = RayQDF;
  static constexpr int kMaxRegs = kLargeRegs;
  static constexpr bool kFusedR2 = true;
  static __device__ __forceinline__ Ray ray(const RayK& K) { return to_qdf(K); }
  static __device__ __forceinline__ void rhs(const Ray& K, df r, df th, df pr, df pth, df& dr,
                                             df& dth, df& dph, df& dpr, df& dpth,
                                             float& twoH) {
    rhs_q_df(K, r, th, pr, pth, dr, dth, dph, dpr, dpth, twoH);
  }
  static constexpr bool kTrackH = true;
  static constexpr bool kF32Stages = false;
  static constexpr double kLocateRel = 4e-16;
  static __device__ __forceinline__ float end_twoH(const Ray& K, const RayK&, const StateDF& y) {
    df dr, dth, dph, dpr, dpth;
    float twoH;
    rhs(K, y.r, y.th, y.pr, y.pth, dr, dth, dph, dpr, dpth, twoH);
    return twoH;
  }
};

template <class Met, int INTEG, bool kLarge>
__global__ void __maxnreg__(kLarge ? Met::kMaxRegs : 255)
    trace_df64_plain(const __grid_constant__ KernelArgs A) {
  trace_body_df<Met, Kernel::kSteal, INTEG>(A);
}

template <class Met, int INTEG, bool kLarge>
__global__ void __maxnreg__(kLarge ? Met::kMaxRegs : 255)
    trace_df64_persistent(const __grid_constant__ KernelArgs A) {
  trace_body_df<Met, Kernel::kPersistent, INTEG>(A);
}

template <class Met, int INTEG, bool kLarge>
static const void* df64_kernel(Kernel kind) {
  return kind == Kernel::kPersistent ? (const void*)trace_df64_persistent<Met, INTEG, kLarge>
                                     : (const void*)trace_df64_plain<Met, INTEG, kLarge>;
}

template <class Met, int INTEG>
static const void* df64_kernel(Kernel kind, int64_t rays, int64_t line) {
  return rays >= line ? df64_kernel<Met, INTEG, true>(kind)
                      : df64_kernel<Met, INTEG, false>(kind);
}

template <class Met>
static const void* df64_kernel(Kernel kind, int integrator, int64_t rays, int64_t line) {
  return integrator == OSIRIS_RKDP45 ? df64_kernel<Met, OSIRIS_RKDP45>(kind, rays, line)
                                     : df64_kernel<Met, OSIRIS_RKCK45>(kind, rays, line);
}

const void* trace_kernel_df64(Kernel kind, int integrator, int spacetime, int64_t rays) {
  return spacetime == OSIRIS_SPACETIME_QMETRIC
             ? df64_kernel<QMetricDF>(kind, integrator, rays, kLargeLaunchQ)
             : df64_kernel<KerrDF>(kind, integrator, rays, kLargeLaunchKerr);
}

}  // namespace osiris_impl
