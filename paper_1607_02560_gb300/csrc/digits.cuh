// The error-free split of the factorisation's updates (see k_nd_tc.cu): digits of a value relative to
// its row's or column's largest, and the sum of the digit products' levels.
#pragma once

namespace lsp {

constexpr int kDigits = 7, kLevels = 7;               // digits per value, weights kept
constexpr int kExpNone = -100000, kExpBad = 1000000;  // all zero; Inf or NaN inside

// Exponent e with |x| < 2^e (kExpNone for zeros and subnormals, kExpBad for Inf and NaN).
__device__ __forceinline__ int exp_of(double x) {
  const int b = (__double2hiint(x) >> 20) & 0x7ff;
  return b == 0 ? kExpNone : b == 0x7ff ? kExpBad : b - 1022;
}
// Digits of x scaled by 2^-e (|x| < 2^e): X = round(x 2^(62 - e)) = sum_t d[t] 512^(6 - t).
__device__ __forceinline__ void digits_of(double x, int e, int (&d)[kDigits]) {
  const long long bits = __double_as_longlong(x);
  const int b = (int)(bits >> 52) & 0x7ff;
  long long X = 0;
  if (b != 0 && e > kExpNone && e < kExpBad) {
    const long long m = (bits & 0xfffffffffffffLL) | 0x10000000000000LL;  // x = m 2^(b - 1075)
    const int sh = b - 1075 + 62 - e;                                     // at most 9
    if (sh >= 0)
      X = m << sh;
    else if (sh > -62)
      X = (m + (1LL << (-sh - 1))) >> -sh;
    if (bits < 0) X = -X;
  }
#pragma unroll
  for (int t = kDigits - 1; t > 0; --t) {
    d[t] = (int)((X + 256) & 511) - 256;
    X = (X - d[t]) >> 9;
  }
  d[0] = (int)X;
}

// sum_l a[l] 2^(-9 l) times 2^ex as a double, |a[l]| < 2^25 integers: put together exactly as one
// 96-bit integer in units of 2^-54, its leading 64 bits rounded once, to nearest, with integer
// operations; values below the normal range become zero, above it infinite.
__device__ __forceinline__ double sum_of(const int (&a)[kLevels], int ex) {
  const long long lo = (long long)a[3] * (1 << 27) + (long long)a[4] * (1 << 18) +
                       (long long)a[5] * (1 << 9) + a[6];
  const long long hi = (long long)a[0] * (1 << 22) + (long long)a[1] * (1 << 13) +
                       (long long)a[2] * 16 + (lo >> 32);
  // two's complement words w2 w1 w0, then the magnitude
  unsigned w0 = (unsigned)lo, w1 = (unsigned)hi, w2 = (unsigned)(hi >> 32);
  const unsigned neg = (unsigned)((int)w2 >> 31);
  w0 ^= neg;
  w1 ^= neg;
  w2 ^= neg;
  asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;"
      : "+r"(w0), "+r"(w1), "+r"(w2)
      : "r"(neg));
  int be = 95 - 54 + 1023 + ex;  // exponent field, less the leading zeros
  if (w2 == 0) {
    w2 = w1;
    w1 = w0;
    w0 = 0;
    be -= 32;
    if (w2 == 0) {
      w2 = w1;
      w1 = 0;
      be -= 32;
    }
  }
  const int lz = __clz((int)w2);
  be -= lz;
  const unsigned uh = __funnelshift_l(w1, w2, lz), ul = __funnelshift_l(w0, w1, lz);
  // 53 bits of the 64-bit mantissa uh ul (top bit at 63), rounded: its top bit adds 1 to the field
  unsigned long long bits = (((unsigned long long)uh << 32) | ul) >> 11;
  bits += ((ul >> 10) & 1) + ((unsigned long long)(unsigned)(be - 1) << 52);
  if (be <= 0 || w2 == 0) bits = 0;
  if (be >= 2047) bits = 0x7ffULL << 52;
  return __longlong_as_double((long long)(bits | ((unsigned long long)(neg & 0x80000000u) << 32)));
}

}  // namespace lsp
