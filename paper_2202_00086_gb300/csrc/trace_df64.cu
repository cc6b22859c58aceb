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
// Two variants, chosen by the launch's rays. Large launches: 128 registers, so
// that four blocks of 128 threads (16 warps) are resident per SM: the
// double-float dependency chains need the extra warps more than they lose to
// the spilled values, which stay in L1 as long as no shared memory is
// reserved (12 x 1024^2 Kerr set, Mrays/s, Cash-Karp: 168 registers (three
// blocks) 14.4, 128: 15.5, 112: 15.4, 96: 15.3, 80: 14.7). Small launches have
// one or two warps per SM sub-partition and last as long as their longest
// chains: no cap (201-231 registers, two blocks per SM), nothing spilled. 128
// registers / no cap, ms:
//   Kerr render  32^2  5.2 / 3.3     100^2  6.3 / 4.0     160^2  7.4 / 5.2
//               256^2  7.8 / 7.1     360^2 11.9 / 10.1    512^2 18.1 / 18.3
//   disk        100^2  4.3 / 2.9     256^2  5.7 / 5.3     400^2  9.3 / 9.5
//   q-metric     64^2  9.0 / 6.3     300^2 17.7 / 15.4    600^2 38.3 / 42.5
//   Dormand-Prince render  64^2  6.3 / 4.2    400^2 14.1 / 13.4    800^2 39.2 / 43.8
//   particles    5,000  1.1 / 0.75  100,000  2.55 / 2.55
// The line lies at 3.5 times the lanes of the uncapped kernels in flight.
constexpr int64_t kLargeLaunch = 7 * 152 * 256 / 2;
constexpr int kLargeRegs = 128;

template <bool kTiny>
struct KerrDF {
  static constexpr bool kTinyRounds = kTiny;
  using Ray = RayDF;
  static constexpr int kMaxRegs = kTiny ? 80 : kLargeRegs;
  static constexpr bool kFusedR2 = true;
  static __device__ __forceinline__ Ray ray(const RayK& K) { return to_df(K); }
  static __device__ __forceinline__ void rhs(const Ray& K, df r, df th, df pr, df pth, df& dr,
                                             df& dth, df& dph, df& dpr, df& dpth,
                                             float& twoH) {
    rhs_df<kTiny>(K, r, th, pr, pth, dr, dth, dph, dpr, dpth, twoH);
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

template <bool kTiny>
struct QMetricDF {
  static constexpr bool kTinyRounds = kTiny;
  using Ray = RayQDF;
  static constexpr int kMaxRegs = kTiny ? 80 : kLargeRegs;
  static constexpr bool kFusedR2 = true;
  static __device__ __forceinline__ Ray ray(const RayK& K) { return to_qdf(K); }
  static __device__ __forceinline__ void rhs(const Ray& K, df r, df th, df pr, df pth, df& dr,
                                             df& dth, df& dph, df& dpr, df& dpth,
                                             float& twoH) {
    rhs_q_df<kTiny>(K, r, th, pr, pth, dr, dth, dph, dpr, dpth, twoH);
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

template <template <bool> class Met, int INTEG>
static const void* df64_kernel(Kernel kind, int64_t rays) {
  if (kind == Kernel::kTinyRound)
    return (const void*)trace_df64_persistent<Met<true>, INTEG, true>;
  return rays >= kLargeLaunch ? df64_kernel<Met<false>, INTEG, true>(kind)
                              : df64_kernel<Met<false>, INTEG, false>(kind);
}

template <template <bool> class Met>
static const void* df64_kernel(Kernel kind, int integrator, int64_t rays) {
  return integrator == OSIRIS_RKDP45 ? df64_kernel<Met, OSIRIS_RKDP45>(kind, rays)
                                     : df64_kernel<Met, OSIRIS_RKCK45>(kind, rays);
}

const void* trace_kernel_df64(Kernel kind, int integrator, int spacetime, int64_t rays) {
  return spacetime == OSIRIS_SPACETIME_QMETRIC ? df64_kernel<QMetricDF>(kind, integrator, rays)
                                               : df64_kernel<KerrDF>(kind, integrator, rays);
}

}  // namespace osiris_impl
