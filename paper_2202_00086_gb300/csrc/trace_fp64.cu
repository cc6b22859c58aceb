// FP64 trace kernels: every operation of the integrator in double precision.
#include <cuda_runtime.h>

#include "trace_kernel.cuh"

namespace osiris_impl {

// Attempts outside the range of ArithFast (arith64.cuh), with plain FP64
// instructions. Out of line, and on copies of its arguments, so that the
// attempt loop keeps its state in registers.
template <class Met>
struct CkArgs {
  RayK K;
  State y, o, d;
  double h, twoH;
};

template <class Met>
__device__ __noinline__ void ck_step_plain(CkArgs<Met>& a) {
  ck_step64<Met>(a.K, a.y, a.h, a.o, a.d, a.twoH);
}

template <class Met>
struct DpArgs {
  RayK K;
  State y, o, d;
  Deriv k1, k7;
  double h;
  bool have_first;  // k1 = f(y) is given
};

template <class Met>
__device__ __noinline__ void dp_step_plain(DpArgs<Met>& a) {
  dp_step64<Met>(a.K, a.y, a.h, a.have_first, a.k1, a.o, a.d, a.k7);
}

template <int INTEG, class Met, bool kLarge>
struct StepperFP64;

// Cash-Karp: every attempt evaluates its six stages.
template <class Met, bool kLarge>
struct StepperFP64<OSIRIS_RKCK45, Met, kLarge> {
  static constexpr double kLocateRel = 0.0;
  static constexpr bool kTrigTable = Met::kTrigTable;
  static constexpr bool kExpLogTable = Met::kExpLogTable;
  struct RayCache {};
  struct LaneCache {};
  static __device__ __forceinline__ void prepare(const RayK&, RayCache&) {}
  static __device__ __forceinline__ void reset(LaneCache&) {}
  static __device__ __forceinline__ void accepted(LaneCache&) {}
  static __device__ __forceinline__ bool attempt(const RayK& K, const RayCache&, LaneCache&,
                                                 const State& y, double h, State& o, State& d,
                                                 double& twoH, double one, double nz) {
    ArithFast<kLarge> ar(one, nz);
    ck_step64<Met>(K, y, h, o, d, twoH, ar);
    if (ar.bad()) {
      CkArgs<Met> a;
      a.K = K;
      a.y = y;
      a.h = h;
      ck_step_plain<Met>(a);
      o = a.o;
      d = a.d;
      twoH = a.twoH;
    }
    return true;
  }
  static __device__ __forceinline__ double twoH(const RayK& K, const State& y) {
    return twoH64<Met>(K, y);
  }
};

// Dormand-Prince: k1 is carried from the previous accepted attempt's seventh
// stage; it is evaluated only when a ray starts or resumes (a warp evaluates
// it when any of its lanes needs it).
template <class Met, bool kLarge>
struct StepperFP64<OSIRIS_RKDP45, Met, kLarge> {
  static constexpr double kLocateRel = 0.0;
  static constexpr bool kTrigTable = Met::kTrigTable;
  static constexpr bool kExpLogTable = Met::kExpLogTable;
  struct RayCache {};
  struct LaneCache {
    Deriv k1, k7;
    bool valid;
  };
  static __device__ __forceinline__ void prepare(const RayK&, RayCache&) {}
  static __device__ __forceinline__ void reset(LaneCache& c) { c.valid = false; }
  static __device__ __forceinline__ void accepted(LaneCache& c) { c.k1 = c.k7; }
  static __device__ __forceinline__ bool attempt(const RayK& K, const RayCache&, LaneCache& c,
                                                 const State& y, double h, State& o, State& d,
                                                 double& twoH, double one, double nz) {
    ArithFast<kLarge> ar(one, nz);
    dp_step64<Met>(K, y, h, c.valid, c.k1, o, d, c.k7, ar);
    if (ar.bad()) {
      DpArgs<Met> a;
      a.K = K;
      a.y = y;
      a.h = h;
      a.k1 = c.k1;
      a.have_first = c.valid;
      dp_step_plain<Met>(a);
      o = a.o;
      d = a.d;
      c.k1 = a.k1;
      c.k7 = a.k7;
    }
    c.valid = true;
    twoH = c.k1.twoH;
    return true;
  }
  static __device__ __forceinline__ double twoH(const RayK& K, const State& y) {
    return twoH64<Met>(K, y);
  }
};

// Two variants of the Kerr kernels, chosen by the launch's rays.
//
// Small launches last as long as their slowest warps' chains of dependent
// instructions: sums on the FP64 unit, no register cap (the compiler takes
// ~195, two blocks of 128 threads per SM). Large ones are bound by the FP64
// unit: sums on the integer pipes where they are cheap there (ArithFast<true>),
// and four blocks per SM to hide the longer chains. Small / large variant, ms:
//   Cash-Karp   render    32^2  12.3 / 15.3     256^2  24.7 / 29.7
//                        360^2  35.2 / 36.3     512^2  57.7 / 56.7
//                        800^2   128 / 110
//               six in a batch  100^2 23.7 / 26.6    200^2 63.1 / 60.0    400^2  207 / 184
//               disk     256^2  18.7 / 20.4     400^2  30.3 / 29.5     600^2  61.3 / 54.0
//   particles   5,000  2.1 / 2.6     100,000  6.6 / 7.0     400,000  21.7 / 20.1
//   Dormand-Prince render 64^2  14.0 / 17.1     400^2  42.6 / 43.1     800^2   135 / 117
// The line lies at five times the lanes that the small variant keeps in
// flight. Caps of 168 registers (three blocks) with either sums lie between
// the two. The q-metric has the small variant only: twice the integer work
// per evaluation, and the large one is 1-5 % slower up to six 400^2 renders.
constexpr int64_t kLargeLaunch = 5 * 152 * 256;

template <int INTEG, class Met, bool kLarge>
__global__ void __maxnreg__(kLarge ? 128 : 255)
    trace_fp64_plain(const __grid_constant__ KernelArgs A) {
  trace_body<StepperFP64<INTEG, Met, kLarge>, Kernel::kSteal>(A);
}

template <int INTEG, class Met, bool kLarge>
__global__ void __maxnreg__(kLarge ? 128 : 255)
    trace_fp64_persistent(const __grid_constant__ KernelArgs A) {
  trace_body<StepperFP64<INTEG, Met, kLarge>, Kernel::kPersistent>(A);
}

template <int INTEG, class Met, bool kLarge>
static const void* fp64_kernel(Kernel kind) {
  return kind == Kernel::kPersistent ? (const void*)trace_fp64_persistent<INTEG, Met, kLarge>
                                     : (const void*)trace_fp64_plain<INTEG, Met, kLarge>;
}

template <class Met, bool kLarge>
static const void* fp64_kernel(Kernel kind, int integrator) {
  return integrator == OSIRIS_RKDP45 ? fp64_kernel<OSIRIS_RKDP45, Met, kLarge>(kind)
                                     : fp64_kernel<OSIRIS_RKCK45, Met, kLarge>(kind);
}

const void* trace_kernel_fp64(Kernel kind, int integrator, int spacetime, int64_t rays) {
  if (spacetime == OSIRIS_SPACETIME_QMETRIC) return fp64_kernel<QMetric, false>(kind, integrator);
  return rays >= kLargeLaunch ? fp64_kernel<KerrMetric, true>(kind, integrator)
                              : fp64_kernel<KerrMetric, false>(kind, integrator);
}

// a b and a + c issued as fused multiply-adds, fma(a, b, -0) and fma(a, 1, c), for
// the probes below. The -0 and 1 come from constant memory, whose values no
// compiler pass may assume, so that the instruction stays a fused multiply-add.
// (The trace kernels take theirs from vector registers, arith64.cuh: an operand
// in constant memory costs the time of a multiply.)
static __constant__ double kFmaNegZero = -0.0;
static __constant__ double kFmaOne = 1.0;

__device__ __forceinline__ double mul_as_fma(double a, double b) {
  double r;
  asm("fma.rn.f64 %0, %1, %2, %3;" : "=d"(r) : "d"(a), "d"(b), "d"(kFmaNegZero));
  return r;
}
__device__ __forceinline__ double add_as_fma(double a, double c) {
  double r;
  asm("fma.rn.f64 %0, %1, %2, %3;" : "=d"(r) : "d"(a), "d"(kFmaOne), "d"(c));
  return r;
}
__device__ __forceinline__ float mul_as_fma(float a, float b) { return a * b; }
__device__ __forceinline__ float add_as_fma(float a, float c) { return a + c; }

// Roofline probes: kProbeChains independent chains of one arithmetic
// operation per thread (OP 0: fused multiply-add a = a b + c, 1: multiply
// a = a b, 2: add a = a + c, 3: the multiply issued as a fused multiply-add
// with a zero addend, 4: the add issued as a fused multiply-add by one), the
// chain step unrolled so that each loop trip
// issues 4 kProbeChains operations back to back. The operands b and c are
// per-thread values, so the compiler cannot hoist or fold them. This
// translation unit is compiled with contraction off, so a multiply or an add
// stays one instruction of the pipe under test.
constexpr int kProbeChains = 16;
constexpr int kProbeBlock = 256;

template <typename T, int OP>
__device__ __forceinline__ T probe_op(T a, T b, T c) {
  if (OP == 0) return fma(a, b, c);
  if (OP == 1) return a * b;
  if (OP == 2) return a + c;
  if (OP == 3) return mul_as_fma(a, b);
  return add_as_fma(a, c);
}

template <typename T, int OP>
__global__ void __launch_bounds__(kProbeBlock) pipe_probe_kernel(double* out, T b0, T c0,
                                                                 int iters) {
  const T t = (T)threadIdx.x * (T)1e-6;
  const T b = b0 + t * (T)1e-3, c = c0 + t;
  T a[kProbeChains];
#pragma unroll
  for (int k = 0; k < kProbeChains; ++k) a[k] = t + (T)k;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int k = 0; k < kProbeChains; ++k) a[k] = probe_op<T, OP>(a[k], b, c);
  }
  T sum = (T)0;
#pragma unroll
  for (int k = 0; k < kProbeChains; ++k) sum += a[k];
  out[(int64_t)blockIdx.x * blockDim.x + threadIdx.x] = (double)sum;
}

template <typename T, int OP>
static int launch_probe_t(int64_t n_threads, int iters, double* out, cudaStream_t s) {
  const int grid = (int)(n_threads / kProbeBlock);
  const T b = (T)0.999999, c = (T)1e-7;
  pipe_probe_kernel<T, OP><<<grid, kProbeBlock, 0, s>>>(out, b, c, iters);
  return (int)cudaGetLastError();
}

template <typename T>
static const void* probe_kernel_t(int op) {
  switch (op) {
    case 0: return (const void*)pipe_probe_kernel<T, 0>;
    case 1: return (const void*)pipe_probe_kernel<T, 1>;
    case 2: return (const void*)pipe_probe_kernel<T, 2>;
    case 3: return (const void*)pipe_probe_kernel<T, 3>;
    default: return (const void*)pipe_probe_kernel<T, 4>;
  }
}

template <typename T>
static int launch_probe_op(int op, int64_t n_threads, int iters, double* out, cudaStream_t s) {
  switch (op) {
    case 0: return launch_probe_t<T, 0>(n_threads, iters, out, s);
    case 1: return launch_probe_t<T, 1>(n_threads, iters, out, s);
    case 2: return launch_probe_t<T, 2>(n_threads, iters, out, s);
    case 3: return launch_probe_t<T, 3>(n_threads, iters, out, s);
    default: return launch_probe_t<T, 4>(n_threads, iters, out, s);
  }
}

int launch_pipe_probe(int precision, int op, int64_t n_threads, int iters, double* out,
                      void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return precision == OSIRIS_FP64 ? launch_probe_op<double>(op, n_threads, iters, out, s)
                                  : launch_probe_op<float>(op, n_threads, iters, out, s);
}

int probe_resident_blocks(int precision, int op, int* blocks_per_sm) {
  const void* fn = precision == OSIRIS_FP64 ? probe_kernel_t<double>(op)
                                            : probe_kernel_t<float>(op);
  return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, kProbeBlock, 0);
}

}  // namespace osiris_impl
