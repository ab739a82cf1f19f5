// FP64 products on the tensor cores for the exchange-correlation contractions.
//
// What bounds them otherwise: GB300's FP64 pipe, 1.06 TFLOP/s, against 0.6
// PFLOP/s of mma.sync bf16 (both measured).  A row of operands is written as
// integers q = rint(v 2^(55 - e)) under the row's common power of two 2^e >
// max |v|, and q as 8 signed digits of 7 bits, |digit| <= 64, which bf16 holds
// exactly.  A product of two digits is at most 2^12, so the FP32 accumulator of
// the tensor core holds the sum of the up to 8 digit products of one weight
// (i + j = k) over 512 terms exactly (8 x 512 x 2^12 = 2^24): no rounding
// happens before the nine sums of weights k = 0..8 are put together, in 64-bit
// integers and one FP64 FMA.  43 bf16 products replace one FP64 product; the
// pairs left out (k > 8) are below 2^-63 of 2^(e_a + e_b) per term, and the
// digits represent an operand to 2^-56 of its row's maximum, where a plain FP64
// sum rounds every step to 2^-53 of its partial sum.
// mma.sync rather than tcgen05: nine accumulators of 128 x N FP32 fill the 512
// columns of TMEM at N = 56, and at such N a tcgen05.mma is bound by reading A
// from shared memory; the register form also takes its A operand as it is
// gathered (digit rows of D at the block's functions) or converted (Z).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace eri {

constexpr int kDigits = 8;        // digits of an operand
constexpr int kWeights = 9;       // digit weights k = i + j kept
constexpr int kExactTerms = 512;  // terms of one exact accumulation

// biased exponent (0 .. 2047) of a double
__device__ __forceinline__ int exponent_of(double v) {
  return (int)((unsigned)__double2hiint(v) >> 20 & 0x7ffu);
}

// The digits of v under the row exponent E = max exponent_of: bf16 of the digits
// in the high halves of d[0] (most significant) .. d[7]
__device__ __forceinline__ void digits_of(double v, int E, uint32_t* d) {
  const long long bits = __double_as_longlong(v);
  const int ex = (int)(bits >> 52) & 0x7ff, r = E - ex - 2;  // q = mantissa 2^-r
  long long m = ex ? ((bits & 0xfffffffffffffLL) | 0x10000000000000LL) : 0LL;
  if (r <= 0) m <<= -r;
  else m = r < 56 ? (m + (1LL << (r - 1))) >> r : 0LL;
  // + 64 in every digit: unsigned digits 0..127 (the top one 0..128)
  constexpr long long kBias = 64LL * 0x2040810204081LL;  // 64 (128^8 - 1) / 127, top digit included
  const unsigned long long u = (unsigned long long)((bits < 0 ? -m : m) + kBias);
#pragma unroll
  for (int i = 0; i < kDigits; ++i) {
    const unsigned x = (unsigned)(u >> (7 * (kDigits - 1 - i))) & (i == 0 ? 0xffu : 0x7fu);
    d[i] = __float_as_uint(__uint_as_float(0x4b000000u | x) - 8388672.0f);  // x - 64, exact in bf16
  }
}
// bf16 pair (k, k + 1) of one digit from two such words
__device__ __forceinline__ uint32_t bf16_pair(uint32_t lo, uint32_t hi) { return __byte_perm(lo, hi, 0x7632); }

// scale of a row with exponent E, so that value = combine() * scale_a * scale_b;
// rows below 2^-960 count as zero
__device__ __forceinline__ double digit_scale(int E) {
  return E > 63 ? __longlong_as_double((long long)(E - 33) << 52) : 0.0;
}

// D[16 x 8] += A[16 x 16] B[16 x 8], bf16 operands, FP32 accumulators
__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, const uint2& b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// the nine exact sums of element c of a tile -> sum 2^(-7 k) s_k, times 2^56
template <int N>
__device__ __forceinline__ double combine(const float (&acc)[kWeights][N], int c) {
  long long hi = 0, lo = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) hi = hi * 128 + __float2int_rn(acc[k][c]);
#pragma unroll
  for (int k = 4; k < kWeights; ++k) lo = lo * 128 + __float2int_rn(acc[k][c]);
  return fma((double)hi, 34359738368.0 /* 2^35 */, (double)lo);
}

}  // namespace eri
