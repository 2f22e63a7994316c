// FP64 products on the integer pipes.
//
// GB300 completes 2 FP64 instructions per clock per SM: one warp instruction occupies a
// sub-partition's FP64 pipe for 64 cycles (measured with 8 warps per sub-partition: 67.5 for a DFMA on
// registers, 81.5 for a DADD or DMUL), while the integer and FP32 pipes stand nearly idle (an
// integer multiply-add costs 2.1 cycles, a logic operation or shift 2.1, a 32 x 32 -> 64 bit multiply-add
// 4 to 6).  The product below is 34 integer instructions, 55 cycles, and runs entirely in
// the shadow of the FP64 pipe: four of them beside four DFMAs take 282 cycles against 276 for
// the DFMAs alone.  So in the kernels bound by that pipe the plain products move here and
// the FP64 pipe keeps the sums and FMAs.  (A sum in integers is 107 cycles: not worth it.)
//
// The product is the IEEE one, rounded to nearest even, bit for bit, for operands and a result that are normal
// numbers: the two 53-bit significands are multiplied exactly as 53 x 64 bits, so that the
// high word pair is the result's significand (53 bits for a product in [2, 4), one bit short in
// [1, 2)) and the low pair its rounding remainder.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ocpg {

// a * b for normal a, b with a normal product; `x` receives the sum of the two exponent fields.
__device__ __forceinline__ double soft_product(double a, double b, uint32_t& x) {
  const uint32_t ah = __double2hiint(a), al = __double2loint(a), bh = __double2hiint(b), bl = __double2loint(b);
  x = (ah & 0x7ff00000u) + (bh & 0x7ff00000u);
  const uint32_t mh = (ah & 0x000fffffu) | 0x00100000u;                                // a: 53 bits
  const uint32_t nh = __funnelshift_l(bl, bh, 11) | 0x80000000u, nl = bl << 11;        // b: 53 bits, left-justified in 64
  const uint64_t t00 = (uint64_t)al * nl;
  const uint64_t t01 = (uint64_t)al * nh + (t00 >> 32);
  const uint64_t t10 = (uint64_t)mh * nl + (uint32_t)t01;
  const uint64_t t11 = (uint64_t)mh * nh + (t01 >> 32) + (t10 >> 32);
  uint32_t h1 = (uint32_t)(t11 >> 32), h0 = (uint32_t)t11;
  uint32_t l = (uint32_t)t10 | min((uint32_t)t00, 1u);     // the remainder's high word, the low one as a sticky bit
  const uint32_t s = (h1 >> 20) ^ 1u;                      // 1: the significands' product is below 2, one more bit comes up
  h1 = __funnelshift_l(h0, h1, s);
  h0 = __funnelshift_l(l, h0, s);
  l = l << s;
  // round to nearest even by the carry out of l + 0x7fffffff + (last bit); the hidden bit of h1 adds
  // one to the exponent field, which is counted in 0x3ff00000 and s
  const uint32_t e = x - 0x3ff00000u - (s << 20) + ((ah ^ bh) & 0x80000000u);
  uint32_t r0, r1;
  asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %2, %3;\n\taddc.cc.u32 %0, %4, 0;\n\taddc.u32 %1, %5, %6;\n\t}"
      : "=r"(r0), "=r"(r1) : "r"(l), "r"(0x7fffffffu + (h0 & 1u)), "r"(h0), "r"(h1), "r"(e));
  return __hiloint2double((int)r1, (int)r0);
}

// Which products may go there.  A node's work runs with integer products if the node's inputs are
// non-zero with 2^-64 <= |v| < 2^64 (soft_input; zeros fill whole vectors at a solver's start
// point, and a warp that holds one does its work with the FP64 pipe's products alone), and is
// done again with those if any product's exponent fields add up to less than 2^-400 or more than
// 2^400 stands for (SoftConst::worst): a zero or subnormal operand (field 0), an infinite or NaN one (field
// 2047) and every product near the ends of the range come out there.  (0 times infinity or NaN
// alone would not: the inputs exclude both, the denominators are tested like inputs, and
// nothing overflows before a product has passed 2^400.)
constexpr uint32_t SOFT_LO = (1023u - 64u) << 20, SOFT_RANGE = 128u << 20;
constexpr uint32_t SOFT_BASE = (2u * 1023u - 400u) << 20, SOFT_SPAN = 800u << 20;
__host__ __device__ __forceinline__ bool soft_input_hi(uint32_t hi) { return (hi & 0x7fffffffu) - SOFT_LO < SOFT_RANGE; }
__device__ __forceinline__ bool soft_input(const double* p) {   // from the high word alone
  return soft_input_hi(__ldg(reinterpret_cast<const uint32_t*>(p) + 1));
}
__device__ __forceinline__ bool soft_value(double v) { return soft_input_hi((uint32_t)__double2hiint(v)); }

}  // namespace ocpg
