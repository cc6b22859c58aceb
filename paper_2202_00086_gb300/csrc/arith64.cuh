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
// fails the test (bad()) is done again with plain FP64 instructions. Factors
// that are zero in ordinary use (the spin of Schwarzschild, L of the middle
// column, p_theta of the middle row) are never given to soft_mul.
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

// Plain FP64 instructions: the end point of a ray, and the attempts that
// ArithFast gives back.
struct ArithPlain {
  __device__ __forceinline__ double mul(double a, double b) const { return a * b; }
  __device__ __forceinline__ double soft(double a, double b) const { return a * b; }
  __device__ __forceinline__ double add(double a, double c) const { return a + c; }
  __device__ __forceinline__ double sub(double a, double c) const { return a - c; }
  __device__ __forceinline__ double unit() const { return 1.0; }
  __device__ __forceinline__ void window(double) const {}
};

struct ArithFast {
  double one, nz;
  unsigned range;  // collects the exponent bits that leave the window

  __device__ __forceinline__ ArithFast(double one_, double nz_)
      : one(one_), nz(nz_), range(0) {}
  // products and sums left on the FP64 unit
  __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, nz); }
  __device__ __forceinline__ double add(double a, double c) const { return fma(a, one, c); }
  __device__ __forceinline__ double sub(double a, double c) const { return fma(a, one, -c); }
  __device__ __forceinline__ double unit() const { return one; }
  // products on the integer pipes
  __device__ __forceinline__ double soft(double a, double b) const { return soft_mul(a, b); }
  // |x| in [2^-63, 2^65): biased exponents 960..1087, so that 64 more have the leading bits 1000
  __device__ __forceinline__ void window(double x) {
    range |= ((unsigned)(bits_of(x) >> 32) + 0x04000000u) ^ 0x40000000u;
  }
  __device__ __forceinline__ bool bad() const { return (range & 0x78000000u) != 0; }
};

}  // namespace osiris_impl
