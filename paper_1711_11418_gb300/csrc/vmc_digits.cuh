// FP64 products on the BF16 tensor cores without rounding: operands as 56-bit
// fixed-point integers (one exponent per row), cut into seven signed 8-bit
// digits, which BF16 holds exactly.  The digit products of equal weight sum
// exactly in the FP32 accumulators of mma.sync while the sums stay below 2^24,
// and a few integer operations make one FP64 number of them.  (Ozaki, Ogita,
// Oishi, Rump, Numer. Algorithms 59, 95, 2012, split operands so; GB300 does
// two FP64 multiply-adds per clock and SM and three orders of magnitude more
// in BF16.)  Users: the elimination of vmc_gj.cuh and the overlap matrix of
// the plain form, vmc_sr_digits.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vmc_dig {

constexpr int NDIG = 7;              // 8-bit digits of an operand
constexpr int NSUM = 8;              // digit sums kept: weights s + u = 0..7
constexpr int NOEXP = -(1 << 20);    // exponent of a group of zeros

// Biased exponent of x (0: zero or subnormal, taken as zero).
__device__ __forceinline__ int expo(double x) {
  return (int)(((unsigned)__double2hiint(x) >> 20) & 0x7ffu);
}

// x 2^(55 - (e - 1022)) rounded to an integer, |q| <= 2^55, for |x| < 2^(e - 1022),
// plus 128 in each of the six lower bytes: digit 0 (weight 2^48) is the value of
// the bits from 48 up, digit s = 1..6 (weight 2^(48 - 8 s)) byte 6 - s less 128.
__device__ __forceinline__ long long fixed(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  const int d = min(max(e - ex, 0), 56);
  long long m = ((b & 0x000fffffffffffffll) | 0x0010000000000000ll) << 2;   // 55 bits
  m = (m + ((1ll << d) >> 1)) >> d;
  if (ex == 0) m = 0;
  return (b < 0 ? -m : m) + 0x0000808080808080ll;
}

// Digit s of v as a float (an integer in [-128, 128], exact in BF16): the byte
// placed under the exponent of 2^23, less 2^23 + 128.
__device__ __forceinline__ float digit(long long v, int s) {
  const unsigned hi = (unsigned)(v >> 32), lo = (unsigned)v;
  if (s == 0) return __int_as_float(0x4B000200 + ((int)hi >> 16)) - 8389120.0f;
  const unsigned w = s <= 2 ? hi : lo;
  const unsigned k = s <= 2 ? 2 - s : 6 - s;
  return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440u + k)) - 8388736.0f;
}
// Digits s of two values as a BF16 pair (exact: the upper halves).
__device__ __forceinline__ uint32_t pair(long long v0, long long v1, int s) {
  return __byte_perm(__float_as_uint(digit(v0, s)), __float_as_uint(digit(v1, s)), 0x7632u);
}

// V 2^x as a double (to nearest, ties away from zero; |V| < 2^62).
__device__ __forceinline__ double scaled(long long V, int x) {
  const unsigned long long s = (unsigned long long)V & 0x8000000000000000ull;
  unsigned long long u = (unsigned long long)(V < 0 ? -V : V);
  const int lz = __clzll((long long)u);
  const int e = 1023 + 63 - lz + x;
  // bit 63 set, half of the last of 53 places added (a carry out of the top
  // reaches the exponent), the leading bit added to the exponent field
  u = ((u << (lz & 63)) + 0x400ull);
  const unsigned long long m = (u >> 11) | (u < 0x400ull ? 0x0020000000000000ull : 0ull);
  unsigned long long b = s | (((unsigned long long)(unsigned)(e - 1) << 52) + m);
  if (V == 0 || e <= 0) b = 0;
  if (V != 0 && e >= 2046) b = s | 0x7ff0000000000000ull;
  return __longlong_as_double((long long)b);
}

// Sum of the digit products, n[d] for s + u = d, in units of 2^(E + F - 54) for
// operands below 2^E and 2^F; d = 6 and 7 round into d = 5.  |n[d]| < 2^24.
__device__ __forceinline__ long long combine(const int (&n)[NSUM]) {
  const int p0 = n[0] * 256 + n[1], p1 = n[2] * 256 + n[3];
  const long long p2 = (long long)n[4] * 256 + (n[5] + (int)(((long long)n[6] * 256 + n[7] + 32768) >> 16));
  return (long long)p0 * 4294967296ll + (long long)p1 * 65536ll + p2;
}
// Exponent of the units above, for operands' biased exponents e and f.
__device__ __forceinline__ int unit_expo(int e, int f) { return e + f - 2 * 1022 - 54; }

// c += a b, one 16 x 8 tile with 16 products each (a row, b column operand).
__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

}  // namespace vmc_dig
