// Lattice index of the resonance-free shift (4 m + 2) pi^2 nearest to x (Sec. 4.1); halves away
// from zero.
#pragma once

#include "lsp_internal.h"

namespace lsp {

// One FP64 operation on the usual path (the FP64 pipe is what bounds the passes over v that call
// this): z = x / (4 pi^2) - 1/2 + 1.5 2^32 holds y = (x / pi^2 - 2) / 4 to 2^-20 in its fraction
// bits while |y| < 2^31, so the nearest integer comes from integer operations. y itself is within
// 2^-20 of what the plain IEEE evaluation gives; next to a half-integer (within 2^-15) and for
// larger y that evaluation decides, with explicit round-to-nearest intrinsics (no contraction into
// fused operations). Measured: the point features of a learned build of 2^20 points 44 -> 28 us.
__device__ __forceinline__ int64_t snap_m(double x) {
  const double z = fma(x, kQuarterInvPi2, 6442450944.0 - 0.5);
  const long long b = __double_as_longlong(z);
  const unsigned frac = (unsigned)b & 0xfffffu;  // units of 2^-20
  if ((int)(b >> 52) == 1023 + 32 && (frac < 0x80000u - 32u || frac > 0x80000u + 32u))
    return (int64_t)((((unsigned long long)b & 0xfffffffffffffULL) + 0x80000u) >> 20) -
           2147483648LL;
  const double y = __dmul_rn(__dsub_rn(__ddiv_rn(x, kPi2), 2.0), 0.25);
  return (int64_t)round(y);
}

}  // namespace lsp
