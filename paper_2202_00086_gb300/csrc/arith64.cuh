// FP64 arithmetic for the FP64 kernels, arranged around GB300's FP64 unit.
//
// Each SM sub-partition has its own FP64 unit, which takes 64 cycles per warp
// instruction whatever the number of active lanes, and 80 cycles unless the
// instruction has three operands in vector registers: a multiply, an add, or
// a fused multiply-add with an operand in a uniform register, in constant
// memory or an immediate (measured per instruction in chains of 8, 16 warps
// per SM: 67 against 80 cycles). A sub-partition issues 64 to 80 instructions
// for the integer and FP32 pipes in that time. So:
//   - multiplies and adds that stay on the FP64 unit are issued as fused
//     multiply-adds, a b = fma(a, b, -0) and a + c = fma(a, 1, c), exact
//     identities of IEEE arithmetic, with -0 and 1 held in vector registers
//     (ArithFast::nz, one; read from shared memory, so that no compiler pass
//     knows their values or that they are the same in every lane);
//   - most products are formed on the integer pipes instead (soft_mul): the
//     correctly rounded product, bit for bit what the FP64 unit gives, in 42
//     cycles of the sub-partition that overlap with the FP64 unit's (two
//     fused multiply-adds and one product take 135 cycles at 8 warps per SM,
//     the time of the two alone; with a native multiply 215).
//
// soft_mul covers finite normal operands whose product is normal. Its callers
// do not test each product: they test that the factors which are not products
// themselves lie in [2^-63, 2^65) (window(), two integer instructions a
// value), from which the range of every product follows; an attempt that
// fails the test (bad()) stops and is done with plain FP64 instructions. Factors
// that are zero in ordinary use (the spin of Schwarzschild, L of the middle
// column, p_theta of the middle row) are never given to soft_mul; those that a
// soft_mul0 takes are tested with window0().
#pragma once
#include <cstdint>

#include "convert.cuh"

namespace osiris_impl {

__device__ __forceinline__ unsigned shift_r(unsigned lo, unsigned hi, unsigned n) {
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, n);
#else
  return (unsigned)((((uint64_t)hi << 32) | lo) >> (n & 31));
#endif
}

// a b, rounded to nearest even, for normal a and b with a normal product; the
// sign and exponent fields add (modulo 2^32, so that the signs multiply).
//
// With the significands A (53 bits) and B 2^10 the 128-bit product lies in
// [2^114, 2^116): shifted left by 2 or 1, its top 64 bits are the 53 of the
// result, and the leading bit of the next word (q1) rounds up. Exactly halfway
// (that word 2^31, nothing below), the last bit is then cleared: rounding up
// an even result sets it, and an odd one has become even.
__device__ __forceinline__ double soft_mul(double a, double b) {
  const uint64_t ia = (uint64_t)bits_of(a), ib = (uint64_t)bits_of(b);
  const unsigned ah = (unsigned)(ia >> 32), bh = (unsigned)(ib >> 32);
  const unsigned a1 = (ah & 0xfffffu) | 0x100000u, b1 = (bh & 0xfffffu) | 0x100000u;
  const uint64_t A = ((uint64_t)a1 << 32) | (unsigned)ia;
  const uint64_t B = (((uint64_t)b1 << 32) | (unsigned)ib) << 10;
#ifdef __CUDA_ARCH__
  const uint64_t h = __umul64hi(A, B);
#else
  const uint64_t h = (uint64_t)(((unsigned __int128)A * B) >> 64);
#endif
  const uint64_t l = A * B;
  const unsigned p3 = (unsigned)(h >> 32), p2 = (unsigned)h, p1 = (unsigned)(l >> 32);
  const unsigned n = (p3 >> 19) + 30;  // 32 - the left shift
  const unsigned q3 = shift_r(p2, p3, n), q2 = shift_r(p1, p2, n), q1 = shift_r(0u, p1, n);
  const bool halfway = ((q1 ^ 0x80000000u) | (unsigned)l) == 0;
  // biased exponents, less the bias, the leading bit in q3 and the 30 in n
  const unsigned e = (ah - a1) + (bh - b1 - (1022u << 20) - (30u << 20)) + (n << 20);
#ifdef __CUDA_ARCH__
  unsigned r2, r3;  // (q3 + e : q2) + (leading bit of q1)
  asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %2, %2;\n\taddc.cc.u32 %0, %3, 0;\n\t"
      "addc.u32 %1, %4, %5;\n\t}"
      : "=r"(r2), "=r"(r3)
      : "r"(q1), "r"(q2), "r"(q3), "r"(e));
  if (halfway) r2 &= ~1u;
  return __hiloint2double((int)r3, (int)r2);
#else
  const uint64_t r = (((uint64_t)(q3 + e) << 32) | q2) + (q1 >> 31);
  return double_of((long long)(halfway ? r & ~(uint64_t)1 : r));
#endif
}

// soft_mul for an `a` that may also be zero (a product of zero keeps the sign
// of the factors'). Four integer instructions more.
__device__ __forceinline__ double soft_mul0(double a, double b) {
  const double r = soft_mul(a, b);
  const long long sign = (bits_of(a) ^ bits_of(b)) & (long long)0x8000000000000000ull;
  const bool zero = ((unsigned)(bits_of(a) >> 32) & 0x7ff00000u) == 0;
  return zero ? double_of(sign) : r;
}

// z 2^(e - 1086) with the sign bit `sign`, rounded to nearest even; the
// leading bit of z is bit 60, 61 or 62, and every bit below the result's last
// that is dropped before z was formed is in its bit 0.
__device__ __forceinline__ double round_sum(uint64_t z, unsigned e, unsigned sign) {
  const unsigned zh = (unsigned)(z >> 32), zl = (unsigned)z;
  const unsigned top = zh >> 29;               // 0: bit 60, 1: bit 61, 2 or 3: bit 62
  const unsigned n = 8 + (top > 2 ? 2 : top);  // bits dropped
  const unsigned q2 = shift_r(zl, zh, n), q3 = zh >> n, q1 = shift_r(0u, zl, n);
  const unsigned x = (q2 & 1u) + 0x7fffffffu;
  const unsigned hi = q3 + ((e + n - 11u) << 20) + sign;  // the leading bit adds one to e
#ifdef __CUDA_ARCH__
  unsigned r2, r3;
  asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %2, %3;\n\taddc.cc.u32 %0, %4, 0;\n\t"
      "addc.u32 %1, %5, 0;\n\t}"
      : "=r"(r2), "=r"(r3)
      : "r"(q1), "r"(x), "r"(q2), "r"(hi));
  return __hiloint2double((int)r3, (int)r2);
#else
  const uint64_t carry = ((uint64_t)q1 + x) >> 32;
  return double_of((long long)((((uint64_t)hi << 32) | q2) + carry));
#endif
}

// s + f, rounded to nearest even, for a normal s and a float f with |f| <
// 2^-10 |s| (f zero or an FP32 denormal: s).
__device__ __forceinline__ double soft_add_small(double s, float f) {
  const unsigned sh = (unsigned)(bits_of(s) >> 32), sl = (unsigned)bits_of(s);
  const unsigned fb = __float_as_uint(f);
  const unsigned e = (sh >> 20) & 0x7ffu, ef = (fb >> 23) & 0xffu;
  // significands with the leading bit at bit 61: s, and f shifted right by
  // the difference d of the exponents; its bits beyond the last go into bit 0
  const unsigned d0 = e - 896u - ef, d = d0 > 63u ? 63u : d0;
  const unsigned m = ef ? (fb & 0x7fffffu) | 0x800000u : 0u;
  const uint64_t x = ((uint64_t)((sh & 0xfffffu) | 0x100000u) << 41) | ((uint64_t)sl << 9);
  const uint64_t v = (uint64_t)m << 38;
  uint64_t y = v >> d;
  if ((y << d) != v) y |= 1;
  const uint64_t flip = (uint64_t)((long long)(int)(sh ^ fb) >> 63);
  const uint64_t z = x + ((y ^ flip) - flip);
  return round_sum(z, e + 1u, sh & 0x80000000u);
}

// x 2^k for an x of at most 53 significant bits and a normal result (or 0).
__device__ __forceinline__ double exact_of(long long x, int k) {
  const uint64_t u = (uint64_t)(x < 0 ? -x : x);
  if (u == 0) return 0.0;
  const int lz = clz64((long long)u);
  const uint64_t m = (u << lz) >> 11;  // the leading bit at bit 52 adds one to the exponent
  return double_of((long long)(((uint64_t)(x < 0) << 63) +
                               ((uint64_t)(1085 - lz + k) << 52) + m));
}

// Plain FP64 instructions: the end point of a ray, and the attempts that
// ArithFast gives back.
struct ArithPlain {
  static constexpr bool kRolledSums = false;
  static constexpr double nz = -0.0;
  __device__ __forceinline__ double mul(double a, double b) const { return a * b; }
  __device__ __forceinline__ double soft(double a, double b) const { return a * b; }
  __device__ __forceinline__ double soft0(double a, double b) const { return a * b; }
  __device__ __forceinline__ double add(double a, double c) const { return a + c; }
  __device__ __forceinline__ double sub(double a, double c) const { return a - c; }
  __device__ __forceinline__ double unit() const { return 1.0; }
  // s + f for a correction f
  __device__ __forceinline__ double add_small(double s, float f) const {
    return s + float_to_double0(f);
  }
  __device__ __forceinline__ double minus_two(double r) const { return r - 2.0; }
  __device__ __forceinline__ bool bad() const { return false; }
  __device__ __forceinline__ void window(double) const {}
  __device__ __forceinline__ void window0(double) const {}
  __device__ __forceinline__ void wide0(double) const {}
};

// a + c on the FP64 unit where a sum on the integer pipes does not apply. Out
// of line: the compiler would otherwise issue it every time and select.
#ifdef __CUDACC__
static __device__ __noinline__ double rare_add(double a, double c) { return a + c; }
#else
static inline double rare_add(double a, double c) { return a + c; }
#endif

// kSums: the sums that are cheap on the integer pipes go there too. That
// takes 36 of an attempt's ~280 FP64 instructions, and makes its chain of
// dependent instructions longer: worth it where enough warps are in flight to
// hide that (kLargeLaunch in trace_fp64.cu).
template <bool kSums>
struct ArithFast {
  static constexpr bool kRolledSums = kSums;  // see rk_attempt64
  double one, nz;
  unsigned range;  // collects the exponent bits that leave the window

  __device__ __forceinline__ ArithFast(double one_, double nz_)
      : one(one_), nz(nz_), range(0) {}
  // products and sums left on the FP64 unit
  __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, nz); }
  __device__ __forceinline__ double add(double a, double c) const { return fma(a, one, c); }
  __device__ __forceinline__ double sub(double a, double c) const { return fma(a, one, -c); }
  __device__ __forceinline__ double unit() const { return one; }
  // Sums on the integer pipes where they are cheap there: a small correction,
  // and differences that are exact (r - 2 is a multiple of the last place of r
  // and no larger than r, so it is a double). Outside their range: native.
  __device__ __forceinline__ double add_small(double s, float f) const {
    if (!kSums) return add(s, float_to_double0(f));
    const int d = (int)(((unsigned)(bits_of(s) >> 52)) & 0x7ffu) - 896 -
                  (int)((__float_as_uint(f) >> 23) & 0xffu);
    if (d < 11) return rare_add(s, float_to_double0(f));
    return soft_add_small(s, f);
  }
  __device__ __forceinline__ double minus_two(double r) const {
    if (!kSums) return sub(r, 2.0);
    const unsigned shift = (unsigned)(bits_of(r) >> 52) - 1023u;  // r in [2^shift, 2^(shift+1))
    if (shift > 52u) return rare_add(r, -2.0);
    const long long m = (bits_of(r) & 0xfffffffffffffll) | 0x10000000000000ll;
    return exact_of(m - (long long)(1ull << (53u - shift)), (int)shift - 52);
  }
  // products on the integer pipes
  __device__ __forceinline__ double soft(double a, double b) const { return soft_mul(a, b); }
  __device__ __forceinline__ double soft0(double a, double b) const { return soft_mul0(a, b); }
  // |x| in [2^-63, 2^65): biased exponents 960..1087, so that 64 more have the leading bits 1000
  __device__ __forceinline__ void window(double x) {
    range |= ((unsigned)(bits_of(x) >> 32) + 0x04000000u) ^ 0x40000000u;
  }
  // the same, or zero
  __device__ __forceinline__ void window0(double x) {
    const unsigned v = ((unsigned)(bits_of(x) >> 32) + 0x04000000u) ^ 0x40000000u;
    range |= (bits_of(x) << 1) == 0 ? 0u : v;
  }
  // |x| in [2^-511, 2^513) or zero, for a factor whose product enters sums only:
  // biased exponents 512..1535, so that 512 more have the leading bit set
  __device__ __forceinline__ void wide0(double x) {
    const unsigned v = ~((unsigned)(bits_of(x) >> 32) + 0x20000000u) & 0x40000000u;
    range |= (bits_of(x) << 1) == 0 ? 0u : v;
  }
  __device__ __forceinline__ bool bad() const { return (range & 0x78000000u) != 0; }
};

}  // namespace osiris_impl
