// FP64 products on the tensor cores for the exchange-correlation contractions.
//
// What bounds them otherwise: GB300's FP64 pipe, 1.06 TFLOP/s (eri_peak_probe), against
// 0.6 PFLOP/s of mma.sync f16 (independent m16n8k16 products on every SM, timed
// apart from the library).  The products are taken by slices, as in Ozaki's scheme
// (Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012): a row of operands is
// written as integers q = rint(v 2^(55 - e)) under the row's common power of two
// 2^e > max |v|, and q as 8 signed digits of 7 bits, |digit| <= 64, which f16 holds
// exactly.  A product of two digits is at most 2^12, so the FP32 accumulator of
// the tensor core holds the sum of the up to 8 digit products of one weight
// (i + j = k) over 512 terms exactly (8 x 512 x 2^12 = 2^24): no rounding
// happens before the nine sums of weights k = 0..8 are put together, in
// integers and rounded once.  43 f16 products replace one FP64 product.
// Accuracy: the digits represent an operand to 2^-56 of its row's maximum, and the
// pairs left out (k > 8, six of weight 9) are together below 2^-60 of 2^(e_a + e_b)
// per term.  That is an absolute bound, about 2^-54 max|a| max|b| per term over the
// rows (of D, of one point's phi, of one function's 32 values of Z or phi): in the
// norm no more than the roundings of a plain FP64 sum (measured rms error of V 9e-16
// to 1.4e-15 with either), but not element by element.  An operand 2^-k of its row's
// maximum keeps 55 - k bits, so a sum that is small because each operand is small
// where the other is large has fewer correct digits than a plain sum would give it:
// of two Gaussians that both peak inside the block, 4 bohr apart (3.8e-6 beside
// products of 1) it is right to 5e-12 of itself, 6 bohr apart (1e-14) to 1e-3; over
// points near one of them only, to 1e-17 at any distance.
// mma.sync rather than tcgen05: nine accumulators of 128 x N FP32 fill the 512
// columns of TMEM at N = 56, and at such N a tcgen05.mma is bound by reading A
// from shared memory; the register form also takes its A operand as it is
// gathered (digit rows of D at the block's functions) or converted (Z).
#pragma once
#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace eri {

constexpr int kDigits = 8;        // digits of an operand
constexpr int kWeights = 9;       // digit weights k = i + j kept
constexpr int kExactTerms = 512;  // terms of one exact accumulation

// biased exponent (0 .. 2047) of a double
__device__ __forceinline__ int exponent_of(double v) {
  return (int)((unsigned)__double2hiint(v) >> 20 & 0x7ffu);
}

// v as an integer under the row exponent E = max exponent_of, 64 added to every
// digit: digit i (0: most significant) + 64 = bits 7 (7 - i) .., 7 bits each, the
// top one 8 (0..128)
__device__ __forceinline__ unsigned long long digits_of(double v, int E) {
  const long long bits = __double_as_longlong(v);
  const int ex = (int)(bits >> 52) & 0x7ff, r = E - ex - 2;  // q = mantissa 2^-r
  long long m = ex ? ((bits & 0xfffffffffffffLL) | 0x10000000000000LL) : 0LL;
  if (r <= 0) m <<= -r;
  else m = r < 56 ? (m + (1LL << (r - 1))) >> r : 0LL;
  constexpr long long kBias = 64LL * 0x2040810204081LL;  // 64 (128^8 - 1) / 127
  return (unsigned long long)((bits < 0 ? -m : m) + kBias);
}
// (x + 1024) halves -> x - 64, both exact
__device__ __forceinline__ uint32_t unbias(uint32_t w) {
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), __half2half2(__ushort_as_half(0x6440)));
  return *reinterpret_cast<const uint32_t*>(&h);
}
// digit i of two values as an f16 pair (u0 in the low half)
__device__ __forceinline__ uint32_t digit_pair(unsigned long long u0, unsigned long long u1, int i) {
  const int s = 7 * (kDigits - 1 - i);
  const uint32_t mask = i == 0 ? 0xffu : 0x7fu;
  return unbias(((uint32_t)(u0 >> s) & mask) | (((uint32_t)(u1 >> s) & mask) << 16) | 0x64006400u);
}
// digits i and i + 1 of one value as an f16 pair
__device__ __forceinline__ uint32_t digit_two(unsigned long long u, int i) {
  const int s = 7 * (kDigits - 1 - i);
  const uint32_t mask = i == 0 ? 0xffu : 0x7fu;
  return unbias(((uint32_t)(u >> s) & mask) | (((uint32_t)(u >> (s - 7)) & 0x7fu) << 16) | 0x64006400u);
}

// D[16 x 8] += A[16 x 16] B[16 x 8], f16 operands, FP32 accumulators
__device__ __forceinline__ void mma_f16(float* c, const uint32_t* a, const uint2& b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// Accumulators of products with at most kShortTerms terms may start at kMagic =
// 1.5 2^23: a sum of at most 2^22 is then the difference of the FP32 words, which
// saves the conversions.
constexpr int kShortTerms = 128;
constexpr float kMagic = 12582912.0f;
constexpr int kMagicBits = 0x4b400000;

// value of element c of a tile whose rows have the exponents Ea (operand a) and Eb:
// the nine exact sums s_k are put together as (hi 2^35 + lo) 2^-56 and rounded
// once, in integers (the FP64 pipe is 30 times slower); values below 2^-1022
// count as zero
template <bool MAGIC>
__device__ __forceinline__ double combine(const float (&acc)[kWeights][4], int c, int Ea, int Eb) {
  int s[kWeights];
#pragma unroll
  for (int k = 0; k < kWeights; ++k)
    s[k] = MAGIC ? __float_as_int(acc[k][c]) - kMagicBits : __float2int_rn(acc[k][c]);
  const long long hi = (long long)(s[0] * 128 + s[1]) * 16384 + (s[2] * 128LL + s[3]);
  const long long lo = ((long long)(s[4] * 128LL + s[5]) * 16384 + (s[6] * 128LL + s[7])) * 128 + s[8];
  unsigned long long l = ((unsigned long long)hi << 35) + (unsigned long long)lo;
  unsigned long long h = (unsigned long long)((hi >> 29) + (lo >> 63)) + (l < (unsigned long long)lo ? 1 : 0);
  // magnitude: two's complement of (h, l) where negative (no branches below: the
  // sums of a tile are put together side by side)
  const unsigned long long sg = (unsigned long long)((long long)h >> 63);
  l ^= sg;
  h ^= sg;
  l -= sg;
  h += (sg & 1) & (l == 0 ? 1ULL : 0ULL);
  const bool up = h != 0;
  const unsigned long long top = up ? h : l, low = up ? l : 0;
  const int n = __clzll((long long)top);
  const int e = (up ? 127 : 63) + Ea + Eb - 1089 - n;  // biased exponent of the leading one
  const unsigned long long m = (top << (n & 63)) | (low >> 1 >> (63 - (n & 63)));
  unsigned long long r = ((unsigned long long)(unsigned)(e - 1) << 52) + (m >> 11) + (m >> 10 & 1);
  r = e >= 2047 ? 0x7ff0000000000000ULL : r;
  r = top == 0 || e <= 0 ? 0ULL : r | (sg & (1ULL << 63));
  return __longlong_as_double((long long)r);
}

// The same value (accumulators started at kMagic, sums of at most 2^20) with three FP64
// operations: hi and lo become doubles as the low bits of 1.5 2^52, the sum is
// rounded once, and the exponents are added to the word.
__device__ __forceinline__ double combine_fp64(const float (&acc)[kWeights][4], int c, int Ea, int Eb) {
  int s[kWeights];
#pragma unroll
  for (int k = 0; k < kWeights; ++k) s[k] = __float_as_int(acc[k][c]) - kMagicBits;
  const long long hi = (long long)(s[0] * 128 + s[1]) * 16384 + (s[2] * 128 + s[3]);
  const long long lo = ((long long)(s[4] * 128 + s[5]) * 16384 + (s[6] * 128 + s[7])) * 128 + s[8];
  constexpr long long kOne = 0x4338000000000000LL;  // 1.5 2^52
  constexpr double kBase = 6755399441055744.0, kTop = kBase * 34359738368.0;
  const double h = fma(__longlong_as_double(kOne + hi), 34359738368.0, -kTop);  // hi 2^35, exact
  const double v = h + (__longlong_as_double(kOne + lo) - kBase);
  const int e = exponent_of(v), f = e + Ea + Eb - 2112;
  const bool zero = e == 0 || f <= 0, inf = f >= 2047;
  const int word = __double2hiint(v), hw = inf ? (word & (int)0x80000000) | 0x7ff00000 : word + (f - e) * 1048576;
  return __hiloint2double(zero ? 0 : hw, zero || inf ? 0 : __double2loint(v));
}

// 16-byte copies from global to shared memory, one group per commit
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {  // at most N groups still in flight
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

}  // namespace eri
