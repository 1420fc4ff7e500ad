// split_fixed.cuh - FP64 products on the FP16 tensor cores, error-free.
//
// The FP64 unit of this part does 2 fused multiply-adds a cycle and SM, the
// tensor cores 1024 FP16 ones (mma.sync): a product of blocks is done on the
// latter by splitting both operands into integer digits (Ozaki, Ogita, Oishi
// and Rump, Numer. Algorithms 59 (2012), with the digits of a common fixed
// point, as in the integer form of Ootomo, Ozaki and Yokota, 2024).
//
// A block's values share one exponent: v = T 2^(E - 1081), E the largest
// biased exponent of the block, |T| < 2^59 an integer (the 53-bit mantissa
// shifted up by 6 and down by the exponent difference: a value within 2^6 of
// the largest keeps every bit, and none is off by more than 2^-59 of the
// largest; a product rounded in FP64 is off by 2^-53 of itself).  T is written in six
// balanced base-1024 digits d_0 .. d_5, |d| <= 512, exact in FP16:
// T = sum d_s 2^(10 (5 - s)).  The product of two values is
//   sum_{i,j} d_i d'_j 2^(100 - 10 (i + j)),
// of which the 21 digit products with i + j <= 5 are formed (the rest is
// below 2^-57 of the largest product).  Those of one diagonal i + j share an
// FP32 accumulator; each digit product is at most 2^18.  Over two k-steps of
// 16 (32 real products) the sums of diagonals 0, 1 and 2 (the latter held in
// two accumulators, of two products and of one) stay within 2^24, so they
// are exact integers whatever the data; for diagonals 3 to 5 a rounding of
// the FP32 sum is below 2^-54 of the sum's terms.  After two k-steps the
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
constexpr int SPLIT_EXP_BIAS = 1081;     // v = T 2^(E - 1081)
constexpr int SPLIT_NONFINITE = 0x7ff;

__device__ __forceinline__ int biased_exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
// the exponent a block scales by: that of a value, subnormals as 1
__device__ __forceinline__ int block_exponent(double2 v) {
  return max(1, max(biased_exponent(v.x), biased_exponent(v.y)));
}

// T + 512 (1 + 2^10 + .. + 2^50): the digits plus 512, each in its 10 bits
__device__ __forceinline__ unsigned long long fixed_biased(double v, int E) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32) | (unsigned)__double2loint(v);
  const int sh = min(E - max(e, 1), 63);
  const long long T = (long long)((m << 6) >> sh);
  const long long s = (long long)(hi >> 31);
  constexpr long long B = 512LL * (1LL + (1LL << 10) + (1LL << 20) + (1LL << 30) + (1LL << 40) + (1LL << 50));
  return (unsigned long long)(((T ^ s) - s) + B);
}

// Digit s of (re, im) as a pair of FP16 values (re in the low half).
__device__ __forceinline__ void split_pair(double re, double im, int E, uint32_t (&w)[SPLIT_DIGITS]) {
  const unsigned long long a = fixed_biased(re, E), b = fixed_biased(im, E);
#pragma unroll
  for (int s = 0; s < SPLIT_DIGITS; ++s) {
    const int p = 10 * (5 - s);
    const uint32_t mask = s == 0 ? 0x7ffu : 0x3ffu;   // the top digit plus 512 may reach 1024
    const uint32_t u = ((uint32_t)(a >> p) & mask) | (((uint32_t)(b >> p) & mask) << 16);
    // 0x6400 + u is the FP16 value 1024 + u (u <= 1024); minus 1536 leaves the digit
    const uint32_t h = u + 0x64006400u, c = 0x66006600u;
    asm("sub.f16x2 %0, %1, %2;" : "=r"(w[s]) : "r"(h), "r"(c));
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
