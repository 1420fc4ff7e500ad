// split_fixed.cuh - FP64 products on the FP16 tensor cores, error-free.
//
// The FP64 unit of this part does 2 fused multiply-adds a cycle and SM, the
// tensor cores 1024 FP16 ones (mma.sync): a product of blocks is done on the
// latter by splitting both operands into integer digits (Ozaki, Ogita, Oishi
// and Rump, Numer. Algorithms 59 (2012), with the digits of a common fixed
// point, as in the integer form of Ootomo, Ozaki and Yokota, 2024).
//
// The values of a row of an operand share one exponent: |v| = T 2^(E - 1080), E
// the largest biased exponent of the row, T < 2^58 an integer (the 53-bit
// mantissa shifted up by 5 and down by the exponent difference: a value within
// 2^5 of the largest keeps every bit, and none is off by more than 2^-57 of the
// largest; a product rounded in FP64 is off by 2^-53 of itself).  T is written in six
// balanced base-1024 digits d_0 .. d_5, |d| <= 512, exact in FP16 (the sign
// goes on every digit; blocks too small for their zeros to shift out, E < 65,
// and those with values that are not finite are left to plain sums):
// T = sum d_s 2^(10 (5 - s)).  The product of two values is
//   sum_{i,j} d_i d'_j 2^(100 - 10 (i + j)),
// of which the 21 digit products with i + j <= 5 are formed.  The rest can
// reach 2^-53.7 of the largest product (every digit at +-512: five products of
// 2^18 on diagonal 6); for digits of random signs its root mean square is about
// 2^-57.  Those of one diagonal i + j share an
// FP32 accumulator; each digit product is at most 2^18.  Over two k-steps of
// 16 (32 real products) the sums of diagonals 0, 1 and 2 (the latter held in
// two accumulators, of two products and of one) stay within 2^24, so they
// are exact integers whatever the data.  Diagonal 3 can reach 1.5 x 2^24 where
// all 32 products have digits near 512 of one sign pattern, i.e. for nearly
// equal values all of one such pattern in both operands; it then rounds, by up
// to 2^-46 of the sum of the terms' magnitudes (32 plain additions: 2^-48).
// Digits of random signs stay 16 standard deviations below 2^24.  Diagonals 4
// and 5 round at 2^-55 of that sum or less.  After two k-steps the
// accumulators are added to 64-bit integers: `hi` in units of diagonal 2,
// `lo` in units of diagonal 5; the result is hi 2^30 + lo, converted to FP64
// with one rounding by integer instructions (four FP64 ones would cost more
// than the whole conversion).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace hb {

constexpr int SPLIT_DIGITS = 6;
constexpr int SPLIT_ACC = 7;             // accumulators: diagonals 0 .. 5, and diagonal 2's third product
constexpr int SPLIT_EXP_BIAS = 1080;     // |v| = T 2^(E - 1080)
constexpr int SPLIT_MIN_EXP = 65;

// the exponent a block scales by: 0 when all is zero (subnormals count as 1);
// integer operations only (a comparison with 0.0 is the FP64 unit's)
__device__ __forceinline__ int block_exponent(double2 v) {
  const unsigned a = (unsigned)__double2hiint(v.x) & 0x7fffffffu, b = (unsigned)__double2hiint(v.y) & 0x7fffffffu;
  const unsigned e = max(a, b) >> 20;
  const unsigned any = a | b | (unsigned)__double2loint(v.x) | (unsigned)__double2loint(v.y);
  return (int)max(e, min(any, 1u));
}
__device__ __forceinline__ bool split_exponent_ok(int e) { return e == 0 || (e >= SPLIT_MIN_EXP && e < 0x7ff); }

// T + 512 (1 + 2^10 + .. + 2^50): the digits plus 512, each in its 10 bits (the
// top one at most 256 + 1); E >= 65, so that zero (read as 2^-1022) shifts out
__device__ __forceinline__ unsigned long long fixed_biased(double v, int E) {
  const unsigned hi = (unsigned)__double2hiint(v);
  const int sh = min(E - (int)((hi >> 20) & 0x7ff), 63);
  const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  constexpr unsigned long long B = 512ULL * (1ULL + (1ULL << 10) + (1ULL << 20) + (1ULL << 30) + (1ULL << 40) + (1ULL << 50));
  return ((m << 5) >> sh) + B;
}

// Digit s of v as a pair of FP16 values (re in the low half); im_flip =
// 0x80000000 negates the imaginary part.  Most of the work is integer logic,
// which this part issues at half the rate of its multiply-adds: the digits are
// cut with one shift a part, a byte permutation and one logic operation, and
// bias and sign go on in one packed FP16 multiply-add.
__device__ __forceinline__ void split_pair(double2 v, int E, uint32_t im_flip, uint32_t (&w)[SPLIT_DIGITS]) {
  const unsigned long long a = fixed_biased(v.x, E), b = fixed_biased(v.y, E);
  // packed +-1 and -+1536
  const uint32_t sg = (((uint32_t)__double2hiint(v.x) >> 16) & 0x8000u) |
                      (((uint32_t)__double2hiint(v.y) ^ im_flip) & 0x80000000u);
  const uint32_t one = 0x3c003c00u ^ sg, off = 0xe600e600u ^ sg;
#pragma unroll
  for (int s = 0; s < SPLIT_DIGITS; ++s) {
    const int p = 10 * (5 - s);
    const uint32_t x = (uint32_t)(a >> p);
    const uint32_t y = p < 16 ? (uint32_t)b << (16 - p) : (uint32_t)(b >> (p - 16));
    // 0x6400 + u is the FP16 value 1024 + u; minus 1536 leaves the digit
    const uint32_t h = (__byte_perm(x, y, 0x7610) & 0x03ff03ffu) | 0x64006400u;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(w[s]) : "r"(h), "r"(one), "r"(off));
  }
}

__device__ __forceinline__ void mma_f16(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The accumulators of one element into hi / lo, and zeroed.
__device__ __forceinline__ void split_flush(float& d0, float& d1, float& d2, float& d3, float& d4, float& d5, float& d2b,
                                            long long& hi, long long& lo) {
  hi += (long long)__float2int_rn(d2) + (long long)__float2int_rn(d2b);
  hi += (long long)__float2int_rn(d1) * 1024;
  hi += (long long)__float2int_rn(d0) * 1048576;
  lo += (long long)__float2int_rn(d5);
  lo += (long long)__float2int_rn(d4) * 1024;
  lo += (long long)__float2int_rn(d3) * 1048576;
  d0 = d1 = d2 = d3 = d4 = d5 = d2b = 0.f;
}

// (hi 2^30 + lo) 2^(50 + ex), rounded once
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int ex) {
  unsigned long long l = (unsigned long long)hi << 30;
  long long t = hi >> 34;
  l += (unsigned long long)lo;
  t += (lo >> 63) + (l < (unsigned long long)lo ? 1 : 0);
  const bool neg = t < 0;
  if (neg) {
    l = ~l + 1;
    t = ~t + (l == 0 ? 1 : 0);
  }
  if (t == 0 && l == 0) return 0.0;
  const int n = t ? __clzll(t) : 64 + __clzll((long long)l);
  unsigned long long m;
  if (n >= 64) m = l << (n - 64);
  else m = n ? ((unsigned long long)t << n) | (l >> (64 - n)) : (unsigned long long)t;
  m = (m >> 11) + ((m >> 10) & 1);   // 53 bits (2^53 when the rounding carries)
  const int q = 75 - n + 50 + ex;    // value = m 2^q
  const int f = q + 1075;            // exponent field of m 2^q, m in [2^52, 2^53)
  double r;
  if (f >= 1 && f <= 2045) r = __longlong_as_double((long long)(((unsigned long long)f << 52) + (m - (1ULL << 52))));
  else r = scalbn((double)(long long)m, q);
  return neg ? -r : r;
}

}  // namespace hb
