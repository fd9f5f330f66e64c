// Lattice index of the resonance-free shift (4 m + 2) pi^2 nearest to x (Sec. 4.1); halves away
// from zero.
#pragma once

#include "lsp_internal.h"

namespace lsp {

// y = (x / pi^2 - 2) / 4 in units of 2^-20, from one FP64 operation (the FP64 pipe is what bounds the
// passes over v): z = x / (4 pi^2) - 1/2 + 1.5 2^32 holds y in its fraction bits while
// |y| < 2^31. Within 2 units of y, and of what the plain IEEE evaluations of y and of (4 m + 2) pi^2
// give; false for larger y and non-finite x.
__device__ __forceinline__ bool lattice_fixed(double x, int64_t* y) {
  const double z = fma(x, kQuarterInvPi2, 6442450944.0 - 0.5);
  const long long b = __double_as_longlong(z);
  *y = (b & 0xfffffffffffffLL) - (1LL << 51);
  return (int)(b >> 52) == 1023 + 32;
}
constexpr int64_t kFixedGuard = 32;  // closer than this the plain evaluation decides

// The nearest integer comes from integer operations; next to a half-integer and for larger y the
// plain evaluation decides, with explicit round-to-nearest intrinsics (no contraction into fused
// operations). Measured: the point features of a learned build of 2^20 points 44 -> 28 us.
__device__ __forceinline__ int64_t snap_m(double x) {
  int64_t f;
  const bool ok = lattice_fixed(x, &f);
  const int64_t half = (f & 0xfffff) - 0x80000;
  if (ok && (half > kFixedGuard || half < -kFixedGuard)) return (f + 0x80000) >> 20;
  const double y = __dmul_rn(__dsub_rn(__ddiv_rn(x, kPi2), 2.0), 0.25);
  return (int64_t)round(y);
}

}  // namespace lsp
