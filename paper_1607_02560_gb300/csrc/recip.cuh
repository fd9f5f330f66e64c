// FP64 reciprocal of a pivot.
#pragma once

namespace lsp {

// 1 / x, less than 0.51 ulp off the exact value: from an FP32 reciprocal r of the leading 24 bits of
// the mantissa m, one step of the geometric series 1 / m = r / (1 - e) = r (1 + e + e^2 + ...), e =
// 1 - m r, cut after e^2 (the third-order Newton, or Halley, iteration for a reciprocal: |e| < 2^-22, so
// the cut costs 2^-66), the exponent by integers. Three FP64 operations where the FP64 division takes
// several times that, on a pipe that is serial for one warp. Zeros, subnormals, infinities, NaN and
// results outside the normal range go to the division.
__device__ __forceinline__ double recip_f64(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int ef = (hi >> 20) & 0x7ff;
  const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, lo);  // in [1, 2)
  const unsigned rb = __float_as_uint(
      1.0f / __uint_as_float(0x3f800000u | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)lo >> 29)));
  const double r0 = __hiloint2double((int)((rb >> 3) + (896u << 20)), (int)(rb << 29));
  const double e = fma(-m, r0, 1.0);
  const double r = fma(r0, fma(e, e, e), r0);  // in [1/2, 1]
  const int rh = __double2hiint(r), fld = (rh >> 20) - (ef - 1023);
  if (ef == 0 || ef == 0x7ff || fld < 1 || fld > 2046) return 1.0 / x;
  return __hiloint2double((hi & 0x80000000) | (fld << 20) | (rh & 0xfffff), __double2loint(r));
}

}  // namespace lsp
