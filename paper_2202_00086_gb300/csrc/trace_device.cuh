// Device side of the backward ray tracer: Hamilton's equations for null
// geodesics in Kerr space-time (Sec. 2.1, Sec. 4.3), adaptive Cash-Karp 4(5)
// steps (Sec. 3.1), the |H| constraint error, stopping surfaces (Sec. 4.1,
// Sec. 5) and the per-ray observables.
//
// Execution model (one ray per lane):
//   Every lane of a warp runs the same loop body each iteration: ONE
//   Cash-Karp attempt from its current state with its own step length.
//   What the lane does with the result depends on its mode:
//     INTEGRATE  accept/reject under the error controller; an accepted step
//                that crosses a stopping surface switches the lane to LOCATE
//     LOCATE     the attempt is a trial step length inside the bracket of the
//                crossing (Illinois-modified regula falsi); on convergence the
//                ray finishes (or, for an equatorial crossing outside the
//                disk, resumes integrating)
//     IDLE       no ray (finished; persistent grids refill it from the queue)
//   So surface location and refills never serialise a warp behind one lane:
//   the expensive part (six evaluations of the equations of motion) is the
//   same instruction stream for every lane.
#pragma once

#include <cstdint>

#include "arith64.cuh"
#include "convert.cuh"
#include "df64.cuh"
#include "explog.cuh"
#include "osiris_internal.h"

namespace osiris_impl {

// ---------------------------------------------------------------------------
// Cash-Karp 4(5) tableau (Cash & Karp 1990, the RKCK45 scheme of Sec. 3.1).
// ---------------------------------------------------------------------------
namespace ck {
constexpr double A21 = 1.0 / 5.0;
constexpr double A31 = 3.0 / 40.0, A32 = 9.0 / 40.0;
constexpr double A41 = 3.0 / 10.0, A42 = -9.0 / 10.0, A43 = 6.0 / 5.0;
constexpr double A51 = -11.0 / 54.0, A52 = 5.0 / 2.0, A53 = -70.0 / 27.0, A54 = 35.0 / 27.0;
constexpr double A61 = 1631.0 / 55296.0, A62 = 175.0 / 512.0, A63 = 575.0 / 13824.0,
                 A64 = 44275.0 / 110592.0, A65 = 253.0 / 4096.0;
// fifth-order weights (propagated solution); stages 2 and 5 have weight 0
constexpr double B1 = 37.0 / 378.0, B3 = 250.0 / 621.0, B4 = 125.0 / 594.0,
                 B6 = 512.0 / 1771.0;
// fifth minus embedded fourth order (error estimate weights), exact rationals
constexpr double D1 = -277.0 / 64512.0, D3 = 6925.0 / 370944.0, D4 = -6925.0 / 202752.0,
                 D5 = -277.0 / 14336.0, D6 = 277.0 / 7084.0;
}  // namespace ck

// Dormand-Prince 5(4) tableau (Dormand & Prince 1980, the RKDP45 scheme of
// Sec. 3.1). Seven stages; the seventh is evaluated at the fifth-order
// solution, so it is the first stage of the next step (first same as last).
namespace dp {
constexpr double A21 = 1.0 / 5.0;
constexpr double A31 = 3.0 / 40.0, A32 = 9.0 / 40.0;
constexpr double A41 = 44.0 / 45.0, A42 = -56.0 / 15.0, A43 = 32.0 / 9.0;
constexpr double A51 = 19372.0 / 6561.0, A52 = -25360.0 / 2187.0, A53 = 64448.0 / 6561.0,
                 A54 = -212.0 / 729.0;
constexpr double A61 = 9017.0 / 3168.0, A62 = -355.0 / 33.0, A63 = 46732.0 / 5247.0,
                 A64 = 49.0 / 176.0, A65 = -5103.0 / 18656.0;
// fifth-order weights = the seventh row; b2 = b7 = 0
constexpr double B1 = 35.0 / 384.0, B3 = 500.0 / 1113.0, B4 = 125.0 / 192.0,
                 B5 = -2187.0 / 6784.0, B6 = 11.0 / 84.0;
// fifth minus embedded fourth order, exact rationals
constexpr double D1 = 71.0 / 57600.0, D3 = -71.0 / 16695.0, D4 = 71.0 / 1920.0,
                 D5 = -17253.0 / 339200.0, D6 = 22.0 / 525.0, D7 = -1.0 / 40.0;
}  // namespace dp

// pi/2 split in two doubles: (PIO2_HI - theta) + PIO2_LO has the sign of
// cos(theta) for theta in (-pi/2, 3pi/2), and equals it to first order near
// the equator.
constexpr double PIO2_HI = 1.5707963267948966;
constexpr double PIO2_LO = 6.123233995736766e-17;
constexpr double TWO_PI = 6.283185307179586;
constexpr double PI_D = 3.141592653589793;

enum : int { MODE_IDLE = 0, MODE_INTEGRATE = 1, MODE_LOCATE = 2, MODE_DONE = 3 };
enum : int { SURF_EQUATOR = 0, SURF_CAPTURE = 1, SURF_ESCAPE = 2 };

struct State {  // evolved coordinates and momenta (t does not feed back; not integrated)
  double r, th, ph, pr, pth;
};

// Per-ray constants of the Hamiltonian (Kerr: a and its products; q-metric:
// q and kap = q (2 + q)).
struct RayK {
  double a, a2, aE, aL, E, L;
  double E2;  // 2E
  double q, kap;
};

// ---------------------------------------------------------------------------
// FP64 sine/cosine and reciprocal with few FP64-pipe instructions.
//
// GB300's FP64 pipe takes one warp instruction per 16 SM cycles (a fused
// multiply-add; a separate multiply or add takes 19), while its FP32, integer
// and shared-memory pipes are nearly idle in this kernel; the helpers below
// move the argument reduction, table look-up, seeds and the small sine/cosine
// corrections onto those pipes and keep only the accuracy-critical FP64
// arithmetic.
//
// sincos_tab: theta = N_k + x, where the node N_k is the double nearest to
// k pi/512 (the node index found in FP32), so that x = theta - N_k is exact
// (Sterbenz) and |x| <= pi/1024 (+ FP32 rounding). sin and cos of the node
// itself (not of k pi/512) come from a per-block shared-memory table filled
// with the library sincos; sin x - x and cos x - 1 from their Taylor series
// (truncation below 0.01 ulp at |x| = 0.0031):
//   sin x - x = x^3 (-1/6 + x^2/120),   cos x - 1 = x^2 (-1/2 + x^2/24),
//   sin theta = (S_k + C_k x) + [C_k (sin x - x) + S_k (cos x - 1)],
//   cos theta = (C_k - S_k x) + [C_k (cos x - 1) - S_k (sin x - x)].
// The bracketed corrections are at most 5e-6 of the result and need only
// ~1e-11 relative accuracy, so they are formed in double-float on the FP32
// pipe from x split into two floats by integer operations; the FP64 pipe does
// x itself, C_k x added to S_k and the correction's two words added on: 7 FP64
// instructions for both results, each within ~1.5 ulp. The table covers theta
// in [-pi/16, 17 pi/16], which holds every ray except one passing almost
// exactly over a pole; outside it the library sincos is used.
// ---------------------------------------------------------------------------
constexpr int kTrigPerPi = 512;                      // nodes per pi
constexpr int kTrigFirst = -kTrigPerPi / 16;         // node index of the first entry
constexpr int kTrigNodes = kTrigPerPi + 2 * (kTrigPerPi / 16) + 1;

struct TrigTable {
  double2 sc[kTrigNodes];  // sin N_k, cos N_k
  float4 scf[kTrigNodes];  // the same as double-float pairs (sin hi, lo, cos hi, lo)
  uint64_t n62[kTrigNodes];  // N_k 2^62 (N_k >= 0)
};

__device__ __forceinline__ TrigTable& trig_table() {
  __shared__ TrigTable table;
  return table;
}

// N_k of table entry i: the double nearest to k pi/512.
__device__ __forceinline__ double trig_node(int i) {
  constexpr double STEP = 3.141592653589793116 / kTrigPerPi;  // exact: pi rounded / 2^9
  return (double)(i + kTrigFirst) * STEP;
}

// Fill the block's table (all threads of the block, before any divergence).
__device__ __forceinline__ void trig_table_init() {
  TrigTable& t = trig_table();
  for (int i = threadIdx.x; i < kTrigNodes; i += blockDim.x) {
    const double n = trig_node(i);
    double s, c;
    sincos(n, &s, &c);
    t.sc[i] = make_double2(s, c);
    const float sh = (float)s, ch = (float)c;
    t.scf[i] = make_float4(sh, (float)(s - (double)sh), ch, (float)(c - (double)ch));
    t.n62[i] = n > 0.0 ? (uint64_t)(n * 0x1p62) : 0;
  }
  __syncthreads();
}

// The block's 1 and -0, the vector operands of ArithFast (arith64.cuh): read
// from shared memory, no compiler pass knows their values.
struct FmaUnits {
  double one, nz;
};

__device__ __forceinline__ volatile FmaUnits& fma_units() {
  __shared__ FmaUnits u;
  return u;
}

// All threads of the block, before any divergence.
__device__ __forceinline__ void fma_units_init() {
  if (threadIdx.x == 0) {
    fma_units().one = 1.0;
    fma_units().nz = -0.0;
  }
  __syncthreads();
}

// The block's copy of the exp/log breakpoint tables (explog.cuh), filled by
// all threads of the block before any divergence.
__device__ __forceinline__ osiris_explog::Tables& explog_table() {
  __shared__ osiris_explog::Tables table;
  return table;
}

__device__ __forceinline__ void explog_table_init() {
  osiris_explog::Tables& t = explog_table();
  for (int i = threadIdx.x; i < osiris_explog::kLogN; i += blockDim.x) {
    if (i < osiris_explog::kExpN) t.t2[i] = osiris_explog::kT2[i];
    t.lg[i] = osiris_explog::kLg[i];
  }
  __syncthreads();
}

// theta - N_k, exact. For theta in [2^-10, 4), where N_k and the last place of
// theta are multiples of 2^-62, on the integer pipes.
__device__ __forceinline__ double node_difference(double th, uint64_t, int i, const ArithPlain&) {
  return th - trig_node(i);
}
template <bool kSums>
__device__ __forceinline__ double node_difference(double th, uint64_t n62, int i,
                                                  const ArithFast<kSums>& ar) {
  if (!kSums) return ar.sub(th, trig_node(i));
  const unsigned shift = (unsigned)((uint64_t)bits_of(th) >> 52) - 1013u;
  if (shift > 11u) return rare_add(th, -trig_node(i));
  const uint64_t m = ((uint64_t)bits_of(th) & 0xfffffffffffffull) | 0x10000000000000ull;
  return exact_of((long long)((m << shift) - n62), -62);
}

// The library's sine and cosine, out of line: inlined, its hundreds of
// instructions lie in the middle of the attempt loop (with the other library
// functions and divisions out of line, and the range tests of exp_tab and
// log_tab on bits: 600^2 q-metric render 167.6 -> 155.5 ms, twelve 640^2 Kerr
// renders 830 -> 824).
#ifdef __CUDACC__
static __device__ __noinline__ double2 rare_sincos(double th) {
#else
static inline double2 rare_sincos(double th) {
#endif
  double s, c;
  sincos(th, &s, &c);
  return make_double2(s, c);
}

template <class A = ArithPlain>
__device__ __forceinline__ void sincos_tab(double th, double& s, double& c, A&& ar = A()) {
  using namespace dfc;
  // nearest node in FP32: 1.5 * 2^23 added to round to an integer
  const float tk = fmaf(to_float_rz(th), (float)(kTrigPerPi / 3.14159265358979323846),
                        12582912.0f);
  const int idx = (__float_as_int(tk) - 0x4B400000) - kTrigFirst;
  if ((unsigned)idx >= (unsigned)kTrigNodes) {  // also NaN / inf
    const double2 sc = rare_sincos(th);
    s = sc.x;
    c = sc.y;
    return;
  }
  const TrigTable& t = trig_table();
  const double2 sc = t.sc[idx];
  const float4 scf = t.scf[idx];
  const double x = node_difference(th, t.n62[idx], idx, ar);  // exact
  // the corrections in double-float
  const df xd = split_df(x);
  const df u = df_sqr(xd);                                                    // x^2
  const df q = df_add_f_u(mk(-I3H, -I3L), __fmul_rn(u.hi, 1.0f / 120.0f));    // -1/6 + x^2/120
  const df ds = df_mul(df_mul(xd, u), q);                                     // sin x - x
  const df cm = df_add_f_u(df_scale(u, -0.5f),
                           __fmul_rn(__fmul_rn(u.hi, u.hi), 1.0f / 24.0f));   // cos x - 1
  const df S = mk(scf.x, scf.y), C = mk(scf.z, scf.w);
  const df corr_s = df_add_u(df_mul(C, ds), df_mul(S, cm));
  const df corr_c = df_sub_u(df_mul(C, cm), df_mul(S, ds));
  s = ar.add_small(fma(sc.y, x, ar.add_small(sc.x, corr_s.hi)), corr_s.lo);
  c = ar.add_small(fma(-sc.x, x, ar.add_small(sc.y, corr_c.hi)), corr_c.lo);
}

// max |H - H0| kept as the bit pattern of a non-negative double: |v| and the
// maximum are integer operations; NaN is ignored like fmax does.
__device__ __forceinline__ void track_abs_H(long long& max_bits, double twoH, double H0) {
  const long long b = __double_as_longlong(fma(0.5, twoH, -H0)) & 0x7fffffffffffffffLL;
  if (b <= 0x7ff0000000000000LL && b > max_bits) max_bits = b;
}

#ifdef __CUDACC__
static __device__ __noinline__ double rare_reciprocal(double d) { return 1.0 / d; }
#else
static inline double rare_reciprocal(double d) { return 1.0 / d; }
#endif

// 1/d: FP32 seed x0 (|x0 d - 1| < 2^-21), then one Newton step with the
// cubic term, x0 (1 + e + e^2) with e = 1 - d x0, relative error e^3 plus
// the final rounding (3 FP64 instructions). Outside the FP32 range: 1/d.
template <class A = ArithPlain>
__device__ __forceinline__ double rcp64(double d, A&& ar = A()) {
  const long long b = __double_as_longlong(d);
  const int e = (int)((b >> 52) & 0x7ff) - 1023 + 127;
  if (e < 2 || e > 252) return rare_reciprocal(d);
  const float f = __int_as_float((int)((b >> 32) & 0x80000000) | (e << 23) |
                                 (int)((b >> 29) & 0x7fffff));
  float rf;
#ifdef __CUDA_ARCH__
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(f));
#else
  rf = 1.0f / f;  // host builds of this header (CPU tests): a correctly rounded seed
#endif
  const double x0 = float_to_double(rf);
  const double eps = fma(-d, x0, ar.unit());
  return fma(x0, fma(eps, eps, eps), x0);
}

// ---------------------------------------------------------------------------
// Hamilton's equations in separated form.
//
// With p_t = -E, p_phi = L, the Kerr Hamiltonian H = 1/2 g^{mu nu} p_mu p_nu
// (Eq. ligH) on the inverse of the metric of Eq. Kerr can be written
//   H = N / (2 Sigma),
//   N = Delta p_r^2 + p_theta^2 + W^2 - P^2 / Delta,
//   P = (r^2 + a^2) E - a L,   W = L / sin(theta) - a E sin(theta).
// Its exact derivatives (no use of H = 0, so the flow is the paper's flow
// everywhere, also off the constraint surface) give, with u = P / Delta,
//   r'       =  Delta p_r / Sigma
//   theta'   =  p_theta / Sigma
//   phi'     =  (W / sin + a u) / Sigma
//   p_r'     =  [ r N / Sigma - (r - 1)(p_r^2 + u^2) + 2 r E u ] / Sigma
//   p_theta' =  cos [ W (L / sin^2 + a E) - a^2 sin N / Sigma ] / Sigma
// which are the component equations of Sec. 2.1 after the common factors
// are collected. One reciprocal of Delta Sigma sin(theta) yields all three
// reciprocals. The outputs are the bracketed terms (the derivatives times
// Sigma) and scale = 1 / Sigma, which the stepper folds into its tableau
// coefficients; products are shared where the algebra allows (Sigma from
// r^2 + a^2 - a^2 sin^2, p_r' as Y + r (X - Y) with X = 2H + 2 E u and
// Y = p_r^2 + u^2, L / sin reused). twoH receives 2H = N / Sigma at the
// evaluation point.
// ---------------------------------------------------------------------------
// With ArithFast every product goes to the integer pipes (those that vanish for
// a = 0 or L = 0 through soft0; window_constants tests K once per attempt).
template <class A = ArithPlain>
__device__ __forceinline__ void rhs64(const RayK& K, double r, double th, double pr, double pth,
                                      double& dr, double& dth, double& dph, double& dpr,
                                      double& dpth, double& twoH, double& scale, A&& ar = A()) {
  double s, c;
  sincos_tab(th, s, c, ar);
  const double ra2 = fma(r, r, K.a2);  // r^2 + a^2
  const double a2s = ar.soft0(K.a2, s);
  const double Delta = fma(r, ar.minus_two(r), K.a2);
  // Sigma = r^2 + a^2 cos^2 = (r^2 + a^2) - a^2 sin^2 (no cancellation: r > a)
  const double Sigma = fma(-a2s, s, ra2);
  const double P = fma(ra2, K.E, -K.aL);
  ar.window(s);
  ar.window(Delta);
  ar.window(Sigma);
  ar.window(P);
  ar.window(pr);
  const double DS = ar.soft(Delta, Sigma);
  const double inv = rcp64(ar.soft(DS, s), ar);
  const double sinv = ar.soft(s, inv);  // 1 / (Delta Sigma)
  const double iSig = ar.soft(Delta, sinv);
  const double iDel = ar.soft(Sigma, sinv);
  const double is = ar.soft(DS, inv);
  const double Lis = ar.soft0(K.L, is);  // L / sin
  const double W = fma(-K.aE, s, Lis);
  const double u = ar.soft(P, iDel);
  const double Dpr = ar.soft(Delta, pr);
  const double N = fma(Dpr, pr, fma(pth, pth, fma(W, W, -ar.soft(P, u))));
  ar.window(N);
  const double NiS = ar.soft(N, iSig);
  // Every derivative carries the factor 1/Sigma; it is returned separately
  // (scale) and folded into the stepper's tableau coefficients.
  dr = Dpr;
  dth = pth;
  dph = fma(W, is, ar.soft0(K.a, u));
  // -dH/dr: (1 - r) Y + r X = Y + r (X - Y), Y = u^2 + p_r^2, X = 2H + 2E u
  const double Y = fma(u, u, ar.soft(pr, pr));
  dpr = fma(r, ar.sub(fma(K.E2, u, NiS), Y), Y);
  // -dH/dtheta: cos (W (L / sin^2 + a E) - a^2 sin 2H)
  const double F = fma(W, fma(Lis, is, K.aE), -ar.soft0(a2s, NiS));
  ar.window(c);
  ar.wide0(F);  // of the order of a^2 where L = 0
  dpth = ar.soft0(F, c);
  scale = iSig;
  twoH = NiS;
}

// ---------------------------------------------------------------------------
// Hamilton's equations on the q-metric (Appendix A, Eq. q-metric, signature
// -+++, m = 1). The metric is diagonal, so with f = 1 - 2/r, D = r^2 - 2r,
// X = 1 + sin^2 / D, k = q (2 + q):
//   g^tt = -f^-(1+q), g^rr = f^(1+q) X^k, g^thth = f^q X^k / r^2,
//   g^phph = f^q / (r^2 sin^2),
// and each derivative is g^{mu mu} times its logarithmic derivative
// (d ln f / dr = 2/D, d ln X / dr = -sin^2 (2r - 2) / (D^2 X),
//  d ln X / dtheta = 2 sin cos / (D X)).
// The powers f^q and X^k come from the table-driven exp and log of
// explog.cuh (about a third of the library's FP64 instructions).
// ---------------------------------------------------------------------------
template <class A = ArithPlain>
__device__ __forceinline__ void rhs_q64(const RayK& K, double r, double th, double pr,
                                        double pth, double& dr, double& dth, double& dph,
                                        double& dpr, double& dpth, double& twoH, double& scale,
                                        A&& ar = A()) {
  scale = 1.0;
  double s, c;
  sincos_tab(th, s, c, ar);
  // four reciprocals (1/D, 1/X, 1/sin^2, 1/(f f^q)) serve every quotient:
  // 1/r = (r - 2)/D, and f = (r - 2)/r keeps its relative accuracy at r -> 2
  const double rm2 = ar.minus_two(r);
  ar.window(r);
  ar.window(rm2);
  ar.window(s);
  ar.window(c);
  ar.window(pr);
  const double iD = rcp64(ar.soft(r, rm2), ar);
  const double ir = ar.soft(rm2, iD);
  const double f = ar.soft(rm2, ir);
  const double s2 = ar.soft(s, s);
  const double is2 = rcp64(s2, ar);
  const double X = fma(s2, iD, ar.unit());
  const double iX = rcp64(X, ar);
  const osiris_explog::Tables& T = explog_table();
  const double fq =
      osiris_explog::exp_tab(ar.mul(K.q, osiris_explog::log_tab(f, T.lg, ar)), T.t2, ar);
  const double Xk =
      osiris_explog::exp_tab(ar.mul(K.kap, osiris_explog::log_tab(X, T.lg, ar)), T.t2, ar);
  ar.window(fq);
  ar.window(Xk);
  ar.window(X);
  const double ir2 = ar.soft(ir, ir);
  const double ffq = ar.soft(f, fq);
  const double fXk = ar.soft(fq, Xk);
  const double gtt = -rcp64(ffq, ar);
  const double grr = ar.soft(f, fXk);
  const double gthth = ar.soft(fXk, ir2);
  const double gpp = ar.soft(ar.soft(fq, ir2), is2);
  dr = ar.soft(grr, pr);
  dth = ar.mul(gthth, pth);
  dph = ar.mul(gpp, K.L);
  // the four terms of 2H
  const double Ht = ar.mul(gtt, ar.mul(K.E, K.E)), Hr = ar.soft(dr, pr), Hth = ar.mul(dth, pth),
               Hph = ar.mul(dph, K.L);
  twoH = ar.add(ar.add(Ht, Hr), ar.add(Hth, Hph));
  // -dH/dr = -1/2 sum_mu (d ln g^mumu / dr) H_mu, collected by logarithmic
  // derivative: -1/2 [(1+q) d ln f (Hr - Ht) + k d ln X (Hr + Hth)
  //                   + (q d ln f - 2/r) (Hth + Hph)]
  const double iDX = ar.soft(iD, iX);
  const double HrHth = ar.add(Hr, Hth);
  const double a1 = fma(-K.q, iD, -iD);  // -(1+q)/D
  // k sin^2 (r-1) / (D^2 X)
  const double a2 = ar.mul(ar.mul(ar.mul(ar.mul(K.kap, s2), ar.sub(r, 1.0)), iD), iDX);
  const double a3 = fma(-K.q, iD, ir);  // 1/r - q/D
  dpr = fma(a1, ar.sub(Hr, Ht), fma(a2, HrHth, ar.mul(a3, ar.add(Hth, Hph))));
  // -dH/dtheta = -1/2 (k d ln X/dtheta (Hr + Hth) - 2 (cos/sin) Hph)
  //            = sin cos (Hph / sin^2 - k (Hr + Hth) / (D X))
  dpth = ar.mul(ar.soft(c, s), fma(ar.mul(-K.kap, iDX), HrHth, ar.mul(Hph, is2)));
}

// Metric policies for the FP64 steppers.
struct KerrMetric {
  static constexpr bool kTrigTable = true;  // rhs64 reads the block's sincos table
  static constexpr bool kExpLogTable = false;
  static constexpr bool kUnitScale = false;
  template <class A>
  static __device__ __forceinline__ void window_constants(const RayK& K, A& ar) {
    ar.window0(K.a);  // and a^2 is zero or in [2^-126, 1): its products are normal, too
    ar.window0(K.L);
  }
  template <class A>
  static __device__ __forceinline__ void rhs(const RayK& K, double r, double th, double pr,
                                             double pth, double& dr, double& dth, double& dph,
                                             double& dpr, double& dpth, double& twoH,
                                             double& scale, A& ar) {
    rhs64(K, r, th, pr, pth, dr, dth, dph, dpr, dpth, twoH, scale, ar);
  }
};
struct QMetric {
  static constexpr bool kTrigTable = true;  // rhs_q64 reads the block's sincos table
  static constexpr bool kExpLogTable = true;  // and the exp/log tables
  static constexpr bool kUnitScale = true;
  template <class A>
  static __device__ __forceinline__ void window_constants(const RayK&, A&) {}
  template <class A>
  static __device__ __forceinline__ void rhs(const RayK& K, double r, double th, double pr,
                                             double pth, double& dr, double& dth, double& dph,
                                             double& dpr, double& dpth, double& twoH,
                                             double& scale, A& ar) {
    rhs_q64(K, r, th, pr, pth, dr, dth, dph, dpr, dpth, twoH, scale, ar);
  }
};

// One evaluation of Hamilton's equations in scaled form: the derivative of
// the evolved components (r, theta, phi, p_r, p_theta) is scale * (r, th, ph,
// pr, pth); twoH = 2H at the evaluation point.
struct Deriv {
  double r, th, ph, pr, pth;
  double scale, twoH;
};

template <class Met = KerrMetric, class A = ArithPlain>
__device__ __forceinline__ void rhs64_at(const RayK& K, double r, double th, double pr,
                                         double pth, Deriv& k, A&& ar = A()) {
  Met::rhs(K, r, th, pr, pth, k.r, k.th, k.ph, k.pr, k.pth, k.twoH, k.scale, ar);
}

template <class Met = KerrMetric, class A = ArithPlain>
__device__ __forceinline__ void rhs64_at(const RayK& K, const State& y, Deriv& k, A&& ar = A()) {
  rhs64_at<Met>(K, y.r, y.th, y.pr, y.pth, k, ar);
}

// 2H at a state (used once per ray for the terminal point).
template <class Met = KerrMetric>
__device__ __forceinline__ double twoH64(const RayK& K, const State& y) {
  Deriv k;
  rhs64_at<Met>(K, y, k);
  return k.twoH;
}

// Embedded Runge-Kutta attempt of length h from y (FP64 everywhere): o =
// fifth-order result, d = fifth minus fourth order. The stage derivative
// k_j = scale_j * k~_j enters every sum through the coefficient
// T.a[s][j] * (h scale_j), so the evaluations never multiply their outputs by
// 1/Sigma; the stage inputs and o are accumulated directly onto y (a few ulp
// of |y| per step, far below the truncation error at any usable tolerance).
// phi is cyclic: its stage values are never needed, only its increment. With
// FSAL the last stage is evaluated at o itself and is the first stage of the
// next step.

// The rows a[s][j], j < s, where the rolled stage loop can index them.
#ifdef __CUDACC__
#define OSIRIS_TABLEAU64 static __constant__
#else
#define OSIRIS_TABLEAU64 static const
#endif
OSIRIS_TABLEAU64 double kCashKarpA[6][6] = {
    {0, 0, 0, 0, 0, 0},
    {ck::A21, 0, 0, 0, 0, 0},
    {ck::A31, ck::A32, 0, 0, 0, 0},
    {ck::A41, ck::A42, ck::A43, 0, 0, 0},
    {ck::A51, ck::A52, ck::A53, ck::A54, 0, 0},
    {ck::A61, ck::A62, ck::A63, ck::A64, ck::A65, 0}};
OSIRIS_TABLEAU64 double kDormandPrinceA[6][6] = {
    {0, 0, 0, 0, 0, 0},
    {dp::A21, 0, 0, 0, 0, 0},
    {dp::A31, dp::A32, 0, 0, 0, 0},
    {dp::A41, dp::A42, dp::A43, 0, 0, 0},
    {dp::A51, dp::A52, dp::A53, dp::A54, 0, 0},
    {dp::A61, dp::A62, dp::A63, dp::A64, dp::A65, 0}};  // the seventh stage is evaluated at o
// The weights b (fifth order) and e (fifth minus embedded fourth order) of both.
OSIRIS_TABLEAU64 double kWeights64[2][2][7] = {
    {{ck::B1, 0, ck::B3, ck::B4, 0, ck::B6, 0}, {ck::D1, 0, ck::D3, ck::D4, ck::D5, ck::D6, 0}},
    {{dp::B1, 0, dp::B3, dp::B4, dp::B5, dp::B6, 0},
     {dp::D1, 0, dp::D3, dp::D4, dp::D5, dp::D6, dp::D7}}};
#undef OSIRIS_TABLEAU64

struct CashKarp64 {
  static constexpr int kStages = 6;
  static constexpr bool kFsal = false;
  static __device__ __forceinline__ double a(int s, int j) { return kCashKarpA[s][j]; }
  static __device__ constexpr double b(int j) {  // fifth-order weights
    constexpr double B[6] = {ck::B1, 0, ck::B3, ck::B4, 0, ck::B6};
    return B[j];
  }
  static __device__ constexpr double e(int j) {  // fifth minus embedded fourth order
    constexpr double E[6] = {ck::D1, 0, ck::D3, ck::D4, ck::D5, ck::D6};
    return E[j];
  }
};

struct DormandPrince64 {
  static constexpr int kStages = 7;
  static constexpr bool kFsal = true;
  static __device__ __forceinline__ double a(int s, int j) { return kDormandPrinceA[s][j]; }
  static __device__ constexpr double b(int j) {
    constexpr double B[7] = {dp::B1, 0, dp::B3, dp::B4, dp::B5, dp::B6, 0};
    return B[j];
  }
  static __device__ constexpr double e(int j) {
    constexpr double E[7] = {dp::D1, 0, dp::D3, dp::D4, dp::D5, dp::D6, dp::D7};
    return E[j];
  }
};

// One attempt. With have_first the first stage is `first`; otherwise it is
// evaluated and returned there. `last` receives the last stage. An attempt that
// leaves the window of ArithFast stops at the next stage, and before the first
// one where its length or the ray's constants do: those fail at every attempt
// of a ray (spins below 2^-63), and a 256^2 render would take the time of both
// attempts (a = 1e-25, Cash-Karp / Dormand-Prince: 43.4 / 48.3 ms against
// 26.3 / 29.6; 20.4 / 21.5 at a = 0). The test costs small Cash-Karp launches
// 0.6 % (64^2 11.04 -> 11.11 ms); large ones and Dormand-Prince ones run 1-2 %
// faster with it.
//
// The stage loop is rolled, with the stage values in local memory (~100
// 8-byte loads per attempt, from L1): one copy of the evaluation keeps the
// loop inside the instruction cache, where six copies with the products on
// the integer pipes do not fit (the q-metric's least of all). Measured with
// plain FP64 multiplies and six copies / products on the integer pipes and
// six copies / and one copy: twelve 320^2 Kerr renders in one launch 338 /
// 267 / 248 ms, a 333 x 257 q-metric render 57.3 / 59.9 / 44.2 ms. The large
// variant (A::kRolledSums) rolls the sums of the result and of the error, too:
// twelve 640^2 renders 857 -> 831 ms; the small one is 4 % slower that way.
template <class Met, class Tab, class A>
__device__ __forceinline__ void rk_attempt64(const RayK& K, const State& y, double h,
                                             bool have_first, Deriv& first, State& o, State& d,
                                             Deriv& last, A& ar) {
  constexpr int NS = Tab::kStages;
  constexpr int NI = Tab::kFsal ? NS - 1 : NS;  // stages whose input is a stage sum
  struct {
    double r, th, ph, pr, pth, w;  // k~_j and w_j = h scale_j
  } k[NS];
  ar.window(h);
  Met::window_constants(K, ar);
  if (have_first) {
    // a kept first stage may come from an attempt with plain instructions
    if (!Met::kUnitScale) ar.window(first.scale);
    k[0] = {first.r, first.th, first.ph, first.pr, first.pth,
            Met::kUnitScale ? h : ar.soft(h, first.scale)};
  }
  // o += b_j w_j k~_j and d += e_j w_j k~_j; a product is the sum with -0
  auto add_result = [&](double b, int j) {
    const double c = ar.soft(b, k[j].w);
    o.r = fma(c, k[j].r, o.r);
    o.th = fma(c, k[j].th, o.th);
    o.ph = fma(c, k[j].ph, o.ph);
    o.pr = fma(c, k[j].pr, o.pr);
    o.pth = fma(c, k[j].pth, o.pth);
  };
  auto add_error = [&](double e, int j) {
    const double c = ar.soft(e, k[j].w);
    d.r = fma(c, k[j].r, d.r);
    d.th = fma(c, k[j].th, d.th);
    d.ph = fma(c, k[j].ph, d.ph);
    d.pr = fma(c, k[j].pr, d.pr);
    d.pth = fma(c, k[j].pth, d.pth);
  };
  auto fifth_order = [&]() {
    o = y;
    if (A::kRolledSums) {
#pragma unroll 1
      for (int j = 0; j < NI; ++j) {
        const double b = kWeights64[Tab::kFsal][0][j];
        if (bits_of(b) != 0) add_result(b, j);
      }
    } else {
#pragma unroll
      for (int j = 0; j < NI; ++j)
        if (Tab::b(j) != 0.0) add_result(Tab::b(j), j);
    }
  };
#pragma unroll 1
  for (int s = have_first ? 1 : 0; s < NS; ++s) {
    if (ar.bad()) return;  // the caller takes plain instructions instead
    double ir = y.r, it = y.th, ip = y.pr, iq = y.pth;
    if (Tab::kFsal && s == NS - 1) {
      fifth_order();
      ir = o.r;
      it = o.th;
      ip = o.pr;
      iq = o.pth;
    } else {
#pragma unroll 1
      for (int j = 0; j < s; ++j) {
        const double c = ar.soft(Tab::a(s, j), k[j].w);
        ir = fma(c, k[j].r, ir);
        it = fma(c, k[j].th, it);
        ip = fma(c, k[j].pr, ip);
        iq = fma(c, k[j].pth, iq);
      }
    }
    Deriv ks;
    rhs64_at<Met>(K, ir, it, ip, iq, ks, ar);
    k[s] = {ks.r, ks.th, ks.ph, ks.pr, ks.pth, Met::kUnitScale ? h : ar.soft(h, ks.scale)};
    if (s == 0) first = ks;
    if (s == NS - 1) last = ks;
  }
  if (!Tab::kFsal) fifth_order();
  d.r = d.th = d.ph = d.pr = d.pth = ar.nz;
  if (A::kRolledSums) {
#pragma unroll 1
    for (int j = 0; j < NS; ++j) {
      const double e = kWeights64[Tab::kFsal][1][j];
      if (bits_of(e) != 0) add_error(e, j);
    }
  } else {
#pragma unroll
    for (int j = 0; j < NS; ++j)
      if (Tab::e(j) != 0.0) add_error(Tab::e(j), j);
  }
}

// One Cash-Karp attempt of length h from y (Sec. 3.1, RKCK45).
template <class Met = KerrMetric, class A = ArithPlain>
__device__ __forceinline__ void ck_step64(const RayK& K, const State& y, double h, State& o,
                                          State& d, double& twoH, A&& ar = A()) {
  Deriv first, last;
  rk_attempt64<Met, CashKarp64>(K, y, h, false, first, o, d, last, ar);
  twoH = first.twoH;
}

// One Dormand-Prince attempt of length h from y (Sec. 3.1, RKDP45): k1 = f(y)
// is given, or evaluated first and returned (have_first = false), then six
// new evaluations; k7 = f(o) is the first stage of the next step if this one
// is accepted.
template <class Met = KerrMetric, class A = ArithPlain>
__device__ __forceinline__ void dp_step64(const RayK& K, const State& y, double h,
                                          bool have_first, Deriv& k1, State& o, State& d,
                                          Deriv& k7, A&& ar = A()) {
  rk_attempt64<Met, DormandPrince64>(K, y, h, have_first, k1, o, d, k7, ar);
}

template <class Met = KerrMetric>
__device__ __forceinline__ void dp_step64(const RayK& K, const State& y, double h,
                                          const Deriv& k1, State& o, State& d, Deriv& k7) {
  Deriv first = k1;
  dp_step64<Met>(K, y, h, true, first, o, d, k7);
}

// True when x is +-inf or NaN (exponent bits all set); integer test only.
__device__ __forceinline__ bool not_finite(double x) {
  return ((__double2hiint(x) >> 20) & 0x7ff) == 0x7ff;
}

__device__ __forceinline__ bool state_not_finite(const State& s) {
  return not_finite(s.r) | not_finite(s.th) | not_finite(s.ph) | not_finite(s.pr) |
         not_finite(s.pth);
}

// Error test of one component: accept needs |d| <= tol (1 + max(|y|, |o|));
// the ratio (for the step-size controller only) is formed in FP32.
__device__ __forceinline__ void err_component(double y, double o, double d, double tol,
                                              bool& ok, float& err) {
  const double scale = tol * (1.0 + fmax(fabs(y), fabs(o)));
  const double ad = fabs(d);
  ok = ok && (ad <= scale);
  err = fmaxf(err, __fdividef((float)ad, (float)scale));
}

// |x| as FP32 by truncating the significand with integer operations only
// (relative error < 2^-23; values below the FP32 normal range become 0,
// above it +inf). Keeps these conversions off the FP64 pipe.
__device__ __forceinline__ float abs_to_float_rz(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
  const int e = (int)(b >> 52) - 1023 + 127;
  if (e <= 0) return 0.0f;
  if (e >= 255) return __int_as_float(0x7f800000);
  return __int_as_float((e << 23) | (int)((b >> 29) & 0x7fffffull));
}

// The error norm of a step (max over the five components of
// |d| / (tol (1 + max(|y|, |o|)))) in FP32 from truncated copies; the ratio is
// within a relative 1e-6 of the FP64 one. The caller decides accept/reject
// from it and falls back to the exact FP64 test (err_component) only when it
// lies within 1e-5 of 1, so the decision is always the FP64 one.
__device__ __forceinline__ float err_norm32(const State& y, const State& o, const State& d,
                                            float tol32) {
  float err = 0.0f;
#define OSIRIS_ERR32(c)                                                                  \
  err = fmaxf(err, __fdividef(abs_to_float_rz(d.c),                                     \
                              tol32 * (1.0f + fmaxf(abs_to_float_rz(y.c),               \
                                                    abs_to_float_rz(o.c)))))
  OSIRIS_ERR32(r);
  OSIRIS_ERR32(th);
  OSIRIS_ERR32(ph);
  OSIRIS_ERR32(pr);
  OSIRIS_ERR32(pth);
#undef OSIRIS_ERR32
  return err;
}

// Value whose sign tells which side of a stopping surface a state is on;
// the crossing is where it changes sign.
__device__ __forceinline__ double surface_value(int kind, const State& s, double r_cap,
                                                double r_esc) {
  if (kind == SURF_EQUATOR) return (PIO2_HI - s.th) + PIO2_LO;  // sign of cos(theta)
  if (kind == SURF_CAPTURE) return s.r - r_cap;
  return s.r - r_esc;
}

// a < b for b > 0 and an a that is not NaN, on the integer pipe.
__device__ __forceinline__ bool less_than_positive(double a, double b) {
  return bits_of(a) < bits_of(b);
}

// An integer that orders as the double does (-0 before 0, NaN outside all):
// the bits of a negative double order backwards, so all but its sign are
// flipped.
__device__ __forceinline__ long long ordered(double x) {
  const long long b = bits_of(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

// The smaller of two values that are not NaN, on the integer pipe.
__device__ __forceinline__ double min_by_bits(double a, double b) {
  return ordered(b) < ordered(a) ? b : a;
}

// The sign of cos(theta) changes between two finite states. theta is a double
// and pi/2 is not, so (PIO2_HI - theta) + PIO2_LO is never zero and is
// positive exactly for theta <= PIO2_HI.
__device__ __forceinline__ bool crosses_equator(const State& y0, const State& y1) {
  return (bits_of(y0.th) <= bits_of(PIO2_HI)) != (bits_of(y1.th) <= bits_of(PIO2_HI));
}

__device__ __forceinline__ const ReqDev* request_of(const KernelArgs& A, int k) {
  return A.reqs ? (A.reqs + k) : &A.single;
}

// Request owning global ray g (largest k with ray_begin <= g).
__device__ __forceinline__ int find_request(const KernelArgs& A, int64_t g) {
  if (A.reqs == nullptr) return 0;
  int lo = 0, hi = A.n_req - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(&A.reqs[mid].ray_begin) <= g)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// Per-lane totals folded into the stats counters when the lane retires.
struct LaneStats {
  unsigned long long rays = 0, acc = 0, rej = 0, root = 0, rhs = 0, fp64_steps = 0;
  unsigned long long status[6] = {0, 0, 0, 0, 0, 0};
  double max_abs_H = 0.0;
};

__device__ __forceinline__ void flush_stats(const KernelArgs& A, LaneStats& S) {
  if (A.stats == nullptr) return;
  const unsigned FULL = 0xffffffffu;
  unsigned long long v[12] = {S.rays, S.acc, S.rej, S.root, S.rhs, S.status[0], S.status[1],
                              S.status[2], S.status[3], S.status[4], S.status[5], S.fp64_steps};
  double mh = S.max_abs_H;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int q = 0; q < 12; ++q) v[q] += __shfl_xor_sync(FULL, v[q], off);
    mh = fmax(mh, __shfl_xor_sync(FULL, mh, off));
  }
  if ((threadIdx.x & 31) == 0) {
    for (int q = 0; q < 11; ++q)
      if (v[q]) atomicAdd(A.stats + q, v[q]);
    if (v[11]) atomicAdd(A.stats + OSIRIS_STAT_FP64_STEPS, v[11]);
    atomicMax(A.stats + OSIRIS_STAT_MAX_ABS_H, (unsigned long long)__double_as_longlong(mh));
  }
}

}  // namespace osiris_impl
