// Step a3 in FP64 for t = 1 builds in 2D and 3D: g_s and g_s * g_s at the offsets of mu_0 - mu_0
// for every shift, by a one-dimensional fast multipole method.
//
// On the lattice s = (4m + 2) pi^2 (Sec. 4.1) the sums of Sec. 3 and 4.2 depend on the
// frequencies only through r = |p|^2 (see k_stage.cu for X_a and the folding of signs):
//   g_f[o](m) = sum_r N_o(r) w_f(r + m),  N_o(r) = n^-d sum_{|p|^2 = r} prod_i X_{|o_i|}(p_i),
//   w_f(l) = (pi^2 (4 l + 2))^-f = (4 pi^2)^-f (l + 1/2)^-f,
// i.e. the potentials (f = 1) and their derivatives (f = 2) of charges N_o(r) at the integers r,
// at the points x = -m - 1/2. The integers are cut into boxes of 128; a box and its two
// neighbours are summed directly (|r + m| < 256: a table of 512 values of w), everything farther
// through a binary tree of boxes: charges interpolated to 20 Chebyshev nodes per box (moments),
// node-to-node products between boxes two or three apart (the nearest source is three half
// widths from the target box' centre, so 20 nodes reach the FP64 rounding level: truncation
// 5.8^-20), and values at the nodes of the leaf boxes interpolated to the points. f = 2 has its
// own node values (kernel 1/x^2) instead of the derivative of the f = 1 interpolant, which would
// lose two digits near the ends of a box.
//
// What bounds it: the FP64 pipe. The sums stage by stage cost 1.5e9 FP64 instructions in stage 1
// and 0.6e9 in stage 2 at 2D n = 1024 with per-point shifts (93 491 of them); here it is 2e8:
// moments depend on n only and are made once per context; 20 200 per box (6900 boxes; 12 500 where
// mirrored nodes share the work, see k_fmm_m2l_box and k_fmm_l2l) for the translations, 970 per
// shift at the end. Fewer nodes or smaller boxes trade these against each other: without the
// mirroring boxes of 64 cost 266e6 + 56e6, of 256 67e6 + 158e6, of 128 133e6 + 90e6.
// Accuracy: rms error of g relative to the largest g of the shift in units of 2^-53, against extended
// precision with the same operations, here (stage by stage, as builds did before): f = 1 2D n = 32
// 0.6 (1.0), 64 0.6 (0.9), 128 0.7 (0.9), 256 0.9 (1.0), 512 1.0 (1.9), 1024 1.3 (2.3), 3D n = 32 0.25
// (0.31), 64 0.27 (0.33); f = 2 2D 0.4 to 0.6 (0.5 to 1.4), 3D 0.7 (0.7 to 0.8). With node values in
// place of differences, the near sources in one pass and charges summed in doubles f = 1 had 0.9 to
// 2.6 in 2D and up to 0.7 in 3D, f = 2 up to 1.1.
// Measured (both stages, GB300; stage by stage before): 2D n = 1024 per-point shifts 3.68 -> 0.30 ms,
// 65 shifts 0.39 -> 0.07 ms, n = 512 0.49 -> 0.105 ms, n = 256 0.155 -> 0.049 ms, n = 128 0.052 ->
// 0.040 ms, 3D n = 64 0.047 -> 0.030 ms (and two launches fewer for the stage lists).
#include <math.h>

#include <algorithm>
#include <vector>

#include "lsp_internal.h"

namespace lsp {
namespace {

constexpr int kLog = kFmmLog, kBox = 1 << kLog;  // integers per leaf box
constexpr int kQ = 20;                     // Chebyshev nodes per box
constexpr int kThreads = 256;
constexpr int kSubLev = 3;                 // a block of the downward pass ends in 2^3 leaf boxes

// The far part of a box is held as its value at the centre and the differences of the 20 node values
// from it: rounding then is relative to how much the far part varies over a box, not to its size (with
// plain node values each level of the tree added the rounding of the whole far part; see the accuracy
// above). The centre is a sum of two doubles: the first holds the total charges of the source boxes
// times a constant each, the second all that is a difference and the rounding of the first on its way
// down the tree. Column kQ of a table is the centre.
constexpr int kH = kQ / 2, kQ1 = kQ + 1, kRows = kQ + 2;  // rows of a box: nodes, centre hi, lo

// Device tables of the plan (doubles): P2M [128][20], M2M [2][20][20], M2L [2][4][20][21]
// (f = 1, 2; offsets -3, -2, 2, 3; values at the nodes less that at the centre; at the centre less a
// constant c near it), the constants c [2][4], the scales of f = 1, 2 at level 0 [2], L2P [20][128],
// near w [512][2], L2L [2][20][21] (less the centre), and for the symmetric pairs (see k_fmm_m2l_box
// and k_fmm_l2l) the half sums and half differences of M2L [2][2][20][10] at offset 2 and of L2L to
// the lower child [2][10][21].
constexpr int kTabP = 0, kTabM = kTabP + kBox * kQ, kTabK = kTabM + 2 * kQ * kQ,
              kTabC = kTabK + 8 * kQ * kQ1, kTabSc = kTabC + 8, kTabE = kTabSc + 2,
              kTabW = kTabE + kQ * kBox, kTabD = kTabW + 4 * kBox * 2,
              kTabKS = kTabD + 2 * kQ * kQ1, kTabMS = kTabKS + 4 * kQ * kH,
              kTabSize = kTabMS + 2 * kH * kQ1;
static_assert(kTabW % 2 == 0, "16-byte aligned");

// s = a + b with its rounding error e.
__device__ __forceinline__ void two_sum(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
// (hi, lo) += x
__device__ __forceinline__ void add2(double& hi, double& lo, double x) {
  double e;
  two_sum(hi, x, hi, e);
  lo += e;
}

template <int D>
struct Cls;  // classes: sorted tuples over {0, 1, 2}, numbered as in the stage tables
template <>
struct Cls<2> {
  static constexpr int NC = 6;
};
template <>
struct Cls<3> {
  static constexpr int NC = 10;
};

// ---- plan (once per context): charges, leaf lists and moments ------------------------------

__device__ __forceinline__ int isqrt_exact(int x) {  // floor(sqrt(x)), 0 <= x < 2^24
  int q = (int)sqrtf((float)x);
  while (q * q > x) --q;
  while ((q + 1) * (q + 1) <= x) ++q;
  return q;
}

// flag[|p|^2] = 1 for every frequency tuple of [0, half]^D (ordered tuples: p ascending).
template <int D>
__global__ void __launch_bounds__(kThreads) k_fmm_flags(int half, uint8_t* __restrict__ flag) {
  const int64_t P = half + 1, total = D == 2 ? P * P : P * P * P;
  for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * kThreads) {
    const int a = (int)(e % P), b = (int)(e / P % P), c = D == 3 ? (int)(e / P / P) : 0;
    if (a <= b && (D == 2 || b <= c)) flag[a * a + b * b + c * c] = 1;
  }
}

// Charges of source s (one warp): the tuples with |p|^2 = r, the last component from the others. The
// lanes look for tuples, then lane c adds class c of each that was found. The rounding of a charge
// stays in every sum made from it, so they are summed in pairs of doubles (X_a and its remainder Xl)
// and rounded once.
template <int D>
__global__ void __launch_bounds__(kThreads) k_fmm_charges(const int32_t* __restrict__ pos, int ns,
                                                          int half, const double* __restrict__ X,
                                                          const double* __restrict__ Xl,
                                                          double inv_n, double* __restrict__ wgt) {
  constexpr int NC = Cls<D>::NC;
  const int P = half + 1, lane = threadIdx.x & 31;
  int ca = 0, cb = 0, cg = 0;  // this lane's class
  {
    int c = 0;
    for (int a = 0; a < 3; ++a)
      for (int b = a; b < 3; ++b)
        for (int g = D == 2 ? 2 : b; g < 3; ++g, ++c)
          if (c == lane) {
            ca = a;
            cb = b;
            cg = g;
          }
  }
  auto x_of = [&](int a, int p) { return make_double2(X[a * P + p], Xl[a * P + p]); };
  auto times = [](double2 x, double2 y) {
    const double h = x.x * y.x;
    return make_double2(h, fma(x.x, y.x, -h) + fma(x.x, y.y, x.y * y.x));
  };
  for (int64_t s = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; s < ns;
       s += ((int64_t)gridDim.x * kThreads) >> 5) {
    const int r = pos[s];
    double hi = 0.0, lo = 0.0;
    const int total = D == 2 ? P : P * P;
    for (int e0 = 0; e0 < total; e0 += 32) {
      const int e = e0 + lane;
      const int p = D == 2 ? e : e / P, q = D == 2 ? 0 : e - p * P;
      const int rest = e < total ? r - p * p - q * q : -1;
      const int z = rest < 0 ? 0 : isqrt_exact(rest);
      unsigned found = __ballot_sync(0xffffffffu, rest >= 0 && z * z == rest && z <= half);
      while (found) {
        const int from = __ffs(found) - 1;
        found &= found - 1;
        const int fp = __shfl_sync(0xffffffffu, p, from), fq = __shfl_sync(0xffffffffu, q, from);
        const int fz = __shfl_sync(0xffffffffu, z, from);
        double2 t = times(x_of(ca, fp), x_of(cb, D == 2 ? fz : fq));
        if (D == 3) t = times(t, x_of(cg, fz));
        add2(hi, lo, t.x);
        lo += t.y;
      }
    }
    if (lane < NC) wgt[s * NC + lane] = (hi + lo) * inv_n;
  }
}

// For 32 integers: which are sources (bit i: 32 w + i) and the sources before them.
__global__ void __launch_bounds__(kThreads) k_fmm_rank(const int32_t* __restrict__ pos, int ns,
                                                       int64_t words, uint2* __restrict__ rank) {
  for (int64_t w = (int64_t)blockIdx.x * kThreads + threadIdx.x; w < words;
       w += (int64_t)gridDim.x * kThreads) {
    int lo = 0, hi = ns;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (pos[mid] < w * 32)
        lo = mid + 1;
      else
        hi = mid;
    }
    unsigned bits = 0;
    for (int s = lo; s < ns && pos[s] < (w + 1) * 32; ++s) bits |= 1u << (pos[s] & 31);
    rank[w] = make_uint2(bits, (unsigned)lo);
  }
}
// Sources below integer x, of nbox leaf boxes.
__device__ __forceinline__ int sources_below(const uint2* __restrict__ rank, int64_t nbox, int64_t x) {
  const int64_t y = x < 0 ? 0 : (x > nbox * kBox ? nbox * kBox : x);
  const uint2 r = __ldg(rank + (y >> 5));
  return (int)r.y + __popc(r.x & ((1u << (int)(y & 31)) - 1u));
}

// Moments of the leaf boxes, q[box][c][k] = sum over the box' sources of N_c(r) L_k(r).
__global__ void __launch_bounds__(kThreads) k_fmm_p2m(const int32_t* __restrict__ pos,
                                                      const double* __restrict__ wgt, int nc,
                                                      const uint2* __restrict__ rank, int64_t nbox,
                                                      const double* __restrict__ tab,
                                                      double* __restrict__ q) {
  const int64_t total = nbox * nc * kQ;
  for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * kThreads) {
    const int k = (int)(e % kQ), c = (int)(e / kQ % nc);
    const int64_t b = e / kQ / nc;
    const int s0 = sources_below(rank, nbox, b * kBox);
    const int s1 = sources_below(rank, nbox, (b + 1) * kBox);
    double acc = 0.0;
    for (int s = s0; s < s1; ++s)
      acc = fma(wgt[(int64_t)s * nc + c], tab[kTabP + (pos[s] & (kBox - 1)) * kQ + k], acc);
    q[e] = acc;
  }
}

// Total charge of every box of every level, the sum of its moments (their interpolation of 1).
__global__ void __launch_bounds__(kThreads) k_fmm_total(const double* __restrict__ q, int64_t n,
                                                        double* __restrict__ q0) {
  for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * kThreads) {
    double hi = 0.0, lo = 0.0;
    for (int k = 0; k < kQ; ++k) add2(hi, lo, q[e * kQ + k]);
    q0[e] = hi + lo;
  }
}

// Moments of the parent boxes of levels l0 .. l1 - 1 from their children (box 2 b + side). The lowest
// levels take a launch each; from where one block covers a level, one block does the rest.
struct Levels {
  int64_t nsb[kFmmLevels], qoff[kFmmLevels];
};
__global__ void __launch_bounds__(kThreads) k_fmm_m2m(double* __restrict__ q,
                                                      const __grid_constant__ Levels t, int l0,
                                                      int l1, int nc,
                                                      const double* __restrict__ tab) {
  for (int l = l0; l < l1; ++l) {
    const double* qc = q + t.qoff[l - 1] * nc * kQ;
    double* qp = q + t.qoff[l] * nc * kQ;
    const int64_t total = t.nsb[l] * nc * kQ;
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * kThreads) {
      const int k = (int)(e % kQ), c = (int)(e / kQ % nc);
      const int64_t b = e / kQ / nc;
      double acc = 0.0;
      for (int side = 0; side < 2; ++side) {
        if (2 * b + side >= t.nsb[l - 1]) break;
        const double* src = qc + ((2 * b + side) * nc + c) * kQ;
        const double* M = tab + kTabM + (side * kQ + k) * kQ;
        for (int i = 0; i < kQ; ++i) acc = fma(M[i], src[i], acc);
      }
      qp[e] = acc;
    }
    __syncthreads();  // one block: its level is complete before the next reads it
  }
}

// ---- one build ---------------------------------------------------------------------------------

using Tree = FmmTree;

// used[box] = 1 for every box that holds a shift, at every level (lists made on the host; the
// per-point policy marks while it compacts its list).
__global__ void __launch_bounds__(kThreads) k_fmm_mark(const int32_t* __restrict__ list,
                                                       const int32_t* __restrict__ count,
                                                       const __grid_constant__ Tree t,
                                                       uint8_t* __restrict__ used,
                                                       int32_t* __restrict__ err) {
  const int64_t cnt = *count;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * kThreads)
    fmm_mark(t, __ldg(list + i), used, err);
}

// Scale of the f-th power's sums at level l.
__device__ __forceinline__ double level_scale(const double* __restrict__ tab, int f, int l) {
  const double p = 1.0 / (double)((int64_t)1 << l);  // exact
  return __ldg(tab + kTabSc + f) * (f ? p * p : p);
}

// Own values of a box from the boxes two or three apart (children of the parent's neighbours;
// offsets -2, 2, 3 of even boxes, -3, -2, 2 of odd ones: indices 0..3 = -3, -2, 2, 3), every level at
// once: they need only the moments. One thread per value, tables and moments through L1. FP64 pipe.
// Measured with the translation downwards (before: a block per box, tables in shared memory, plain node
// values): 2D n = 32 17.3 -> 15.2 us, 3D n = 64 29.6 -> 25.1 us.
template <int NC>
__global__ void __launch_bounds__(kThreads) k_fmm_m2l(const __grid_constant__ Tree t,
                                                             const uint8_t* __restrict__ used,
                                                             const double* __restrict__ tab,
                                                             const double* __restrict__ q,
                                                             const double* __restrict__ q0,
                                                             double* __restrict__ loc) {
  constexpr int FC = 2 * NC, OUT = FC * kQ1;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, u = e / OUT;
  if (u >= t.off[t.L + 1] || !used[u]) return;
  const int o = (int)(e - u * OUT), i = o / FC, fc = o - i * FC, c = fc >> 1, f = fc & 1;
  int l = 0;
  while (u >= t.off[l + 1]) ++l;
  const int64_t j = t.jlo[l] + (u - t.off[l]);
  double acc[3] = {0.0, 0.0, 0.0}, tot = 0.0;  // three chains side by side
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int di = d + 1 - (int)(j & 1);
    const int64_t x = j + (di < 2 ? di - 3 : di);
    if (x < 0 || x >= t.nsb[l]) continue;
    const double* K = tab + kTabK + ((f * 4 + di) * kQ) * kQ1 + i;
    const double* qq = q + (t.qoff[l] + x) * (NC * kQ) + c * kQ;
    if (i == kQ)
      tot = fma(__ldg(tab + kTabC + f * 4 + di), __ldg(q0 + (t.qoff[l] + x) * NC + c), tot);
#pragma unroll
    for (int k = 0; k < kQ; ++k) acc[d] = fma(__ldg(K + k * kQ1), __ldg(qq + k), acc[d]);
  }
  const double sc = level_scale(tab, f, l), dif = (acc[0] + acc[1] + acc[2]) * sc;
  double* out = loc + u * (FC * kRows) + o;
  if (i < kQ) {
    out[0] = dif;
  } else {
    out[0] = tot * sc;
    out[FC] = dif;
  }
}

constexpr int kBoxThreads = 256;
// The same, a block per box and a thread per pair of mirrored nodes (i, 19 - i). With R the moments
// of the box at offset 2 and L those at -2 in reverse order, K_-2[k][i] = -+K_2[19 - k][19 - i] (f = 1,
// 2) gives
//   out[i] + out[19 - i] = sum_k (K_2[k][i] + K_2[k][19 - i]) (R -+ L)[k],
//   out[i] - out[19 - i] = sum_k (K_2[k][i] - K_2[k][19 - i]) (R +- L)[k],
// 80 instead of 120 multiply-adds a pair with the third offset. The values at the centre by a warp of
// their own where the block has one to spare (any block size will do), in 2D on two lanes a column
// (offsets +-2 and 3): an FP64 instruction of a warp takes 64 cycles of its quarter of the SM, which a
// pair's warp shares. Measured with the translation downwards, plain node values: 2D n = 1024 208 ->
// 175 us, n = 512 53.7 -> 50.0 us, n = 128 20.5 -> 18.7 us.
template <int NC>
__global__ void __launch_bounds__(kThreads) k_fmm_m2l_box(
    const __grid_constant__ Tree t, const uint8_t* __restrict__ used,
    const double* __restrict__ tab, const double* __restrict__ q, const double* __restrict__ q0,
    double* __restrict__ loc) {
  constexpr int FC = 2 * NC, PAIRS = FC * kH;
  __shared__ double sa[2][NC][kQ], s3[NC][kQ];  // R + L, R - L; the moments at offset 3 or -3
  const int64_t boxes = t.off[t.L + 1];
  const int spare = (PAIRS + 31) / 32, warps = blockDim.x >> 5;
  int l = 0;
  for (int64_t u = blockIdx.x; u < boxes; u += gridDim.x) {
    if (!used[u]) continue;
    while (u >= t.off[l + 1]) ++l;
    const int64_t j = t.jlo[l] + (u - t.off[l]);
    const int odd = (int)(j & 1);
    auto inside = [&](int64_t x) { return x >= 0 && x < t.nsb[l]; };
    for (int e = threadIdx.x; e < NC * kQ; e += blockDim.x) {
      const int c = e / kQ, k = e % kQ;
      auto moment = [&](int64_t x, int kk) {
        return inside(x) ? __ldg(q + (t.qoff[l] + x) * (NC * kQ) + c * kQ + kk) : 0.0;
      };
      const double r = moment(j + 2, k), m = moment(j - 2, kQ - 1 - k);
      sa[0][c][k] = r + m;
      sa[1][c][k] = r - m;
      s3[c][k] = moment(odd ? j - 3 : j + 3, k);
    }
    __syncthreads();
    double* out = loc + u * (FC * kRows);
    for (int e = threadIdx.x; e < PAIRS; e += blockDim.x) {
      const int i = e / FC, fc = e - i * FC, c = fc >> 1, f = fc & 1;
      const double* KS = tab + kTabKS + 2 * f * kQ * kH + i;
      const double* K3 = tab + kTabK + ((f * 4 + (odd ? 0 : 3)) * kQ) * kQ1 + i;
      const double *ps = sa[1 - f][c], *pd = sa[f][c], *p3 = s3[c];
      double sum = 0.0, dif = 0.0, lo = 0.0, hi = 0.0;
#pragma unroll
      for (int k = 0; k < kQ; ++k) {
        sum = fma(__ldg(KS + k * kH), ps[k], sum);
        dif = fma(__ldg(KS + (kQ + k) * kH), pd[k], dif);
        lo = fma(__ldg(K3 + k * kQ1), p3[k], lo);
        hi = fma(__ldg(K3 + k * kQ1 + kQ - 1 - 2 * i), p3[k], hi);
      }
      const double sc = level_scale(tab, f, l);
      out[i * FC + fc] = (lo + (sum + dif)) * sc;
      out[(kQ - 1 - i) * FC + fc] = (hi + (sum - dif)) * sc;
    }
    if ((int)(threadIdx.x >> 5) == (warps > spare ? spare : (int)(u % warps))) {
      constexpr bool SPLIT = 2 * FC <= 32;
      const int lane = threadIdx.x & 31, fc = lane % FC, c = fc >> 1, f = fc & 1;
      auto total = [&](int64_t x) {
        return inside(x) ? __ldg(q0 + (t.qoff[l] + x) * NC + c) : 0.0;
      };
      const double ql = total(j - 2), q2 = total(j + 2) + (f ? ql : -ql);  // c at -2 is -+ c at 2
      const double q3 = total(odd ? j - 3 : j + 3);
      const double* K2 = tab + kTabK + ((f * 4 + 2) * kQ) * kQ1 + kQ;
      const double* K3 = tab + kTabK + ((f * 4 + (odd ? 0 : 3)) * kQ) * kQ1 + kQ;
      const double *ps = sa[1 - f][c], *p3 = s3[c];
      double dif = 0.0;
      if (SPLIT) {
        const double *K = lane < FC ? K2 : K3, *p = lane < FC ? ps : p3;
#pragma unroll
        for (int k = 0; k < kQ; ++k) dif = fma(__ldg(K + k * kQ1), p[k], dif);
        dif += __shfl_down_sync(0xffffffffu, dif, FC);
      } else {
#pragma unroll
        for (int k = 0; k < kQ; ++k)
          dif = fma(__ldg(K3 + k * kQ1), p3[k], fma(__ldg(K2 + k * kQ1), ps[k], dif));
      }
      if (lane < FC) {
        const double sc = level_scale(tab, f, l);
        const double tot = fma(__ldg(tab + kTabC + f * 4 + (odd ? 0 : 3)), q3,
                               __ldg(tab + kTabC + f * 4 + 2) * q2);
        out[kQ * FC + fc] = tot * sc;
        out[kQ1 * FC + fc] = dif * sc;
      }
    }
    __syncthreads();  // the next box
  }
}

// Values of the leaves: from the top, child = own + interpolation of the parent's (the centre as one
// more node, its two doubles added to the parent's). A block follows the path to one box of level
// S <= 3, then the boxes below it: S = 3 repeats the least of the upper levels' work (2D n = 1024: 50e6
// FP64 instructions, S = 0 183e6), smaller S spreads a small tree over more SMs (2D n = 128, 55 leaves:
// both passes 40 -> 25 us).
// FS of the 2 NC columns (class, f) per block (they are independent of each other): all, or a quarter
// with S = 0.
template <int NC, int FS>
__global__ void __launch_bounds__(kThreads) k_fmm_l2l(const __grid_constant__ Tree t,
                                                      const uint8_t* __restrict__ used,
                                                      const double* __restrict__ tab,
                                                      double* __restrict__ loc, int S) {
  constexpr int FC = 2 * NC, ALL = FC * kRows, OUT = FS * kQ, OUT1 = FS * kQ1;
  const int f0 = blockIdx.y * FS;
  auto at = [&](int64_t u, int o) {  // place of value o of this block's columns of box u
    return u * ALL + o / FS * FC + f0 + o % FS;
  };
  __shared__ double sM[2 * kQ * kQ1], sS[2 * kH * kQ1];
  __shared__ double buf[2][(1 << (kSubLev - 1)) * OUT];  // levels S - 1.. 1 at most 4 boxes
  __shared__ double2 cen[2][(1 << (kSubLev - 1)) * FS];  // their centres
  const int64_t root = blockIdx.x;  // box of level S
  if (t.L == 0 || !used[t.off[S] + root]) return;
  for (int e = threadIdx.x; e < 2 * kQ * kQ1; e += kThreads) sM[e] = tab[kTabD + e];
  for (int e = threadIdx.x; e < 2 * kH * kQ1; e += kThreads) sS[e] = tab[kTabMS + e];
  const int64_t jr = t.jlo[S] + root;
  // value o of a child: its own (loaded before the parent's part is formed) plus x from the parent;
  // into box b of the next buffer, or memory
  struct Own {
    int64_t g;
    double v, lo;
  };
  auto own = [&](int64_t u, int o) {
    const int64_t g = at(u, o);
    return Own{g, loc[g], o < OUT ? 0.0 : loc[g + FC]};
  };
  auto put = [&](const Own& w, int o, double x, double2 pc, int l, int nx, int b) {
    if (o < OUT) {
      const double v = w.v + x;
      if (l == 0)
        loc[w.g] = v;
      else
        buf[nx][b * OUT + o] = v;
    } else {
      double hi = w.v, lo = w.lo + pc.y;
      add2(hi, lo, pc.x);
      lo += x;
      if (l == 0) {
        loc[w.g] = hi;
        loc[w.g + FC] = lo;
      } else {
        cen[nx][b * FS + (o - OUT)] = make_double2(hi, lo);
      }
    }
  };
  // from the parent's differences src to those of a child on the given side
  auto down = [&](const double* src, int side, int o) -> double {
    const int i = o / FS, fc = o - i * FS;
    const double* M = sM + side * kQ * kQ1 + i;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < kQ; ++k) acc = fma(M[k * kQ1], src[k * FS + fc], acc);
    return acc;
  };
  int cur = 0;
  {
    const int64_t u = t.off[t.L] + (jr >> (t.L - S)) - t.jlo[t.L];
    for (int o = threadIdx.x; o < OUT1; o += kThreads) {
      if (o < OUT)
        buf[0][o] = loc[at(u, o)];
      else
        cen[0][o - OUT] = make_double2(loc[at(u, o)], loc[at(u, o) + FC]);
    }
  }
  auto box = [&](int l) { return t.off[l] + (jr >> (l - S)) - t.jlo[l]; };  // of the path
  if constexpr (FS < FC) {
    // S = 0: only the path, many levels one after the other (65 shifts at 2D n = 1024: eleven), each
    // bound by the latency of a chain of 20 multiply-adds. The centres go to a warp of their own, four
    // lanes each, so that they end with the nodes, and the next level's own values are on their way.
    constexpr int BASE = (OUT + 31) / 32 * 32;
    static_assert(BASE + 32 <= kThreads && 4 * FS <= 32, "one warp");
    const bool node = (int)threadIdx.x < OUT, centre = threadIdx.x >= BASE && threadIdx.x < BASE + 32;
    const int fc = min((int)(threadIdx.x - BASE) >> 2, FS - 1), part = threadIdx.x & 3;
    const int o = node ? threadIdx.x : centre ? OUT + fc : 0;
    Own w = own(box(t.L - 1), o);
    __syncthreads();
    for (int l = t.L - 1; l >= 0; --l, cur ^= 1) {
      const Own next = own(box(l > 0 ? l - 1 : 0), o);
      const int side = (int)(jr >> l) & 1;
      if (node) {
        put(w, o, down(buf[cur], side, o), make_double2(0.0, 0.0), l, cur ^ 1, 0);
      } else if (centre) {
        const double* M = sM + side * kQ * kQ1 + kQ;
        double x = 0.0;
#pragma unroll
        for (int k = 0; k < kQ / 4; ++k)
          x = fma(M[(part + 4 * k) * kQ1], buf[cur][(part + 4 * k) * FS + fc], x);
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        x += __shfl_xor_sync(0xffffffffu, x, 2);
        if ((int)threadIdx.x < BASE + 4 * FS && part == 0) put(w, o, x, cen[cur][fc], l, cur ^ 1, 0);
      }
      w = next;
      __syncthreads();
    }
    return;
  }
  __syncthreads();
  for (int l = t.L - 1; l >= S; --l, cur ^= 1) {
    const int side = (int)(jr >> (l - S)) & 1;
    for (int o = threadIdx.x; o < OUT1; o += kThreads) {
      const Own w = own(box(l), o);
      put(w, o, down(buf[cur], side, o), cen[cur][o % FS], l, cur ^ 1, 0);
    }
    __syncthreads();
  }
  // All columns: both children of a parent together. With e, o the sums and differences of its values
  // at mirrored nodes, node i of the lower child is E + O and node 19 - i of the upper one E - O (the
  // centre mirrors itself), E = sum_k<10 Ms[k][i] e[k], O = sum Md[k][i] o[k]: half the multiply-adds
  // for one more barrier a level (2D n = 1024, both translations, plain node values 216 -> 208 us; with
  // few subtrees the barrier costs more: 3D n = 64 21.4 -> 23.5 us).
  for (int l = S - 1; l >= 0; --l, cur ^= 1) {
    const int np = 1 << (S - 1 - l);  // parents under the root
    double* par = buf[cur];
    for (int e = threadIdx.x; e < np * kH * FS; e += kThreads) {
      const int b = e / (kH * FS), o = e - b * (kH * FS), kk = o / FS, fc = o - kk * FS;
      double* x = par + b * OUT + kk * FS + fc;
      double* y = par + b * OUT + (kQ - 1 - kk) * FS + fc;
      const double vx = *x, vy = *y;
      *x = vx + vy;
      *y = vx - vy;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < np * OUT1; e += kThreads) {
      const int b = e / OUT1, o = e - b * OUT1, i = o / FS, fc = o - i * FS;
      const int64_t x = (jr << (S - l)) + 2 * b - t.jlo[l], u = t.off[l] + x;  // the lower child
      const bool lower = x >= 0 && u < t.off[l + 1] && used[u];
      const bool upper = x + 1 >= 0 && u + 1 < t.off[l + 1] && used[u + 1];
      if (!lower && !upper) continue;
      const double* src = par + b * OUT + fc;
      const int om = i < kQ ? (kQ - 1 - i) * FS + fc : o;  // the mirrored node
      const Own wl = lower ? own(u, o) : Own{0, 0.0, 0.0};
      const Own wu = upper ? own(u + 1, om) : Own{0, 0.0, 0.0};
      double E = 0.0, O = 0.0;
#pragma unroll
      for (int k = 0; k < kH; ++k) {
        E = fma(sS[k * kQ1 + i], src[k * FS], E);
        O = fma(sS[(kH + k) * kQ1 + i], src[(kQ - 1 - k) * FS], O);
      }
      const double2 pc = cen[cur][b * FS + fc];
      if (lower) put(wl, o, E + O, pc, l, cur ^ 1, 2 * b);
      if (upper) put(wu, om, E - O, pc, l, cur ^ 1, 2 * b + 1);
    }
    __syncthreads();
  }
}

struct EvalArgs {
  const int32_t* list;
  const int32_t* count;
  const int32_t* pos;
  const double* wgt;
  const uint2* rank;
  const double* tab;
  const double* loc;
  int64_t jlo, nbox, nsb;
  double* g;
  int64_t cap;
  int32_t* err;
};

// The near sources' terms on top of the far part's differences in acc: this lane has nl sources below
// the point and nr above it, numbered from the far end (source 0 the farthest, at(side, k)), and takes
// those of each side in that order but the nearest of both sides last. So the large terms are rounded
// once: in one pass across the point each term after the nearest was rounded at its size (f = 1 at 2D
// n = 256: the near sums' rms error 1.0 -> 0.5 units of 2^-53 of the largest g).
template <int NC, int UNROLL, class At>
__device__ __forceinline__ void near_sources(const EvalArgs& a, int64_t m, int nl, int nr,
                                             const At& at, double (&acc)[2 * NC]) {
  const double2* sW = reinterpret_cast<const double2*>(a.tab + kTabW);
  const int la = nl > 0 ? nl - 1 : 0, ra = nr > 0 ? nr - 1 : 0;
#pragma unroll UNROLL
  for (int t = 0; t < nl + nr; ++t) {
    const bool tail = t >= la + ra;
    const bool left = tail ? t == la + ra && nl > 0 : t < la;
    const int s = at(left, left ? (tail ? la : t) : (tail ? ra : t - la));
    const double2 w = __ldg(sW + (int)(__ldg(a.pos + s) + m) + 2 * kBox);
    const double2* q = reinterpret_cast<const double2*>(a.wgt + (int64_t)s * NC);
#pragma unroll
    for (int c = 0; c < NC / 2; ++c) {
      const double2 n = __ldg(q + c);
      acc[4 * c] = fma(n.x, w.x, acc[4 * c]);
      acc[4 * c + 1] = fma(n.x, w.y, acc[4 * c + 1]);
      acc[4 * c + 2] = fma(n.y, w.x, acc[4 * c + 2]);
      acc[4 * c + 3] = fma(n.y, w.y, acc[4 * c + 3]);
    }
  }
}

// g = centre + (sum + its low part)
template <int NC>
__device__ __forceinline__ double with_centre(const double* lo, int c, double sum) {
  return __ldg(lo + kQ * 2 * NC + c) + (sum + __ldg(lo + kQ1 * 2 * NC + c));
}

// Differences of the far part at point tp of its leaf box, over nodes lane, lane + lanes, ...
template <int NC>
__device__ __forceinline__ void far_nodes(const EvalArgs& a, const double* lo, int tp, int lane,
                                          int lanes, double (&acc)[2 * NC]) {
  const double* sE = a.tab + kTabE;
#pragma unroll
  for (int c = 0; c < 2 * NC; ++c) acc[c] = 0.0;
  for (int i = lane; i < kQ; i += lanes) {
    const double e = __ldg(sE + i * kBox + tp);
    const double2* v = reinterpret_cast<const double2*>(lo + i * 2 * NC);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const double2 q = __ldg(v + c);
      acc[2 * c] = fma(q.x, e, acc[2 * c]);
      acc[2 * c + 1] = fma(q.y, e, acc[2 * c + 1]);
    }
  }
}

// The sums of N columns over the lanes of a group, O its half. While N is even a lane hands half of its
// columns to its partner and adds what it gets for the others, so it adds N / 2 + N / 4 + .. times
// instead of N times a step. The first columns_left<N, O>() of v hold columns from c0 on.
template <int N, int O>
constexpr int columns_left() {
  if constexpr (O == 0)
    return N;
  else
    return columns_left<(N % 2 == 0 ? N / 2 : N), O / 2>();
}
template <int N, int O, int FC>
__device__ __forceinline__ void group_sum(double (&v)[FC], int lane, int& c0) {
  if constexpr (O > 0 && N % 2 == 0) {
    const bool up = (lane & O) != 0;
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      const double keep = up ? v[k + N / 2] : v[k], send = up ? v[k] : v[k + N / 2];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
    if (up) c0 += N / 2;
    group_sum<N / 2, O / 2>(v, lane, c0);
  } else if constexpr (O > 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], O);
    group_sum<N, O / 2>(v, lane, c0);
  }
}

// g values of every shift, LANES threads per shift: 2 for long lists (2D n = 1024: 1, 2, 4, 8 lanes
// 250, 243, 252, 327 us; one lane leaves too few warps, more repeat the far part's loads and the
// reduction), 8 for short ones (2D n = 256: 68, 38, 30, 30 us; n = 128: 75, 42, 28, 20 us). The
// tables are read through L1 (28 KiB). In 2D 64 registers, so that the 16 blocks of 64 threads of the
// default shape are resident together (2D n = 1024 with 86 registers 232 us, now 200 us).
template <int NC, int LANES>
__global__ void __launch_bounds__(kThreads, NC == 6 ? 4 : 2) k_fmm_eval(EvalArgs a) {
  constexpr int FC = 2 * NC, LEFT = columns_left<FC, LANES / 2>();
  constexpr int SAME = LANES * LEFT / FC;  // lanes that end with the same columns
  const int64_t cnt = *a.count;
  const int lane = threadIdx.x % LANES;
  const int64_t step = (int64_t)gridDim.x * (blockDim.x / LANES);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x / LANES) + threadIdx.x / LANES;
       __any_sync(0xffffffffu, i < cnt); i += step) {
    const bool live = i < cnt;
    const int64_t m = __ldg(a.list + (live ? i : 0));
    const int64_t x = -m, j = x >> kLog, b = checked(j - a.jlo, a.nbox, a.err);
    const double* lo = a.loc + b * (FC * kRows);
    const int s0 = sources_below(a.rank, a.nsb, (j - 1) * kBox);
    const int s1 = sources_below(a.rank, a.nsb, (j + 2) * kBox);
    const int sx = sources_below(a.rank, a.nsb, x);
    double acc[FC];
    far_nodes<NC>(a, lo, (int)(x & (kBox - 1)), lane, LANES, acc);
    near_sources<NC, 2>(
        a, m, (sx - s0 - lane + LANES - 1) / LANES, (s1 - sx - lane + LANES - 1) / LANES,
        [&](bool left, int k) { return left ? s0 + lane + k * LANES : s1 - 1 - lane - k * LANES; },
        acc);
    int c0 = 0;
    group_sum<FC, LANES / 2>(acc, lane, c0);
    if (live && lane % SAME == 0) {
#pragma unroll
      for (int k = 0; k < LEFT; ++k)
        a.g[(int64_t)(c0 + k) * a.cap + i] = with_centre<NC>(lo, c0 + k, acc[k]);
    }
  }
}

// Few shifts: a block of 128 threads (all four FP64 quarters of an SM) per shift. The sources of a
// side go to the threads by their distance from the point, thread 127 the nearest, and the 128 partial
// sums of each value are added by eight lanes, 16 each with the nearest last, then across them with
// the rounding errors carried along.
constexpr int kEvalBlock = 128;
template <int NC>
__global__ void __launch_bounds__(kEvalBlock) k_fmm_eval_block(EvalArgs a) {
  constexpr int FC = 2 * NC;
  __shared__ double part[FC][kEvalBlock + 1];
  const int64_t cnt = *a.count;
  const int tid = threadIdx.x, rank = kEvalBlock - 1 - tid;
  for (int64_t i = blockIdx.x; i < cnt; i += gridDim.x) {
    const int64_t m = __ldg(a.list + i);
    const int64_t x = -m, j = x >> kLog, b = checked(j - a.jlo, a.nbox, a.err);
    const double* lo = a.loc + b * (FC * kRows);
    const int s0 = sources_below(a.rank, a.nsb, (j - 1) * kBox);
    const int s1 = sources_below(a.rank, a.nsb, (j + 2) * kBox);
    const int sx = sources_below(a.rank, a.nsb, x);
    double acc[FC];
    far_nodes<NC>(a, lo, (int)(x & (kBox - 1)), tid, kEvalBlock, acc);
    const int nl = (sx - s0 - rank + kEvalBlock - 1) / kEvalBlock;
    const int nr = (s1 - sx - rank + kEvalBlock - 1) / kEvalBlock;
    near_sources<NC, 4>(
        a, m, nl, nr,
        [&](bool left, int k) {
          return left ? sx - 1 - rank - (nl - 1 - k) * kEvalBlock
                      : sx + rank + (nr - 1 - k) * kEvalBlock;
        },
        acc);
#pragma unroll
    for (int c = 0; c < FC; ++c) part[c][tid] = acc[c];
    __syncthreads();
    const int sub = tid & 7;
    for (int c = tid >> 3; c < (FC + 15) / 16 * 16; c += kEvalBlock / 8) {
      double s = 0.0, e = 0.0;
      if (c < FC)
        for (int k = sub; k < kEvalBlock; k += 8) s += part[c][k];
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const double t = __shfl_xor_sync(0xffffffffu, s, o);
        const double te = __shfl_xor_sync(0xffffffffu, e, o);
        add2(s, e, t);
        e += te;
      }
      if (c < FC && sub == 0) a.g[(int64_t)c * a.cap + i] = with_centre<NC>(lo, c, s + e);
    }
    __syncthreads();
  }
}

int grid_for(int64_t work, int per_block = kThreads) {
  const int64_t b = (work + per_block - 1) / per_block;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

// Host tables in extended precision: L_k at x is (1/Q) (1 + 2 sum_p T_p(s_k) T_p(x)).
std::vector<double> make_tables() {
  typedef long double R;
  const R pi = 3.14159265358979323846264338327950288L;
  std::vector<R> node(kQ);
  for (int k = 0; k < kQ; ++k) node[k] = cosl((2 * k + 1) * pi / (2 * kQ));
  auto cheb = [](R x, R* T) {
    T[0] = 1;
    T[1] = x;
    for (int p = 2; p < kQ; ++p) T[p] = 2 * x * T[p - 1] - T[p - 2];
  };
  std::vector<R> Tn(kQ * kQ);
  for (int k = 0; k < kQ; ++k) cheb(node[k], &Tn[k * kQ]);
  auto basis = [&](R x, R* out) {
    R T[kQ];
    cheb(x, T);
    for (int k = 0; k < kQ; ++k) {
      R s = 0.5L;
      for (int p = 1; p < kQ; ++p) s += Tn[k * kQ + p] * T[p];
      out[k] = 2 * s / kQ;
    }
  };
  std::vector<double> t(kTabSize);
  R b[kQ], bc[kQ];
  for (int i = 0; i < kBox; ++i) {  // source at integer i of its box: (i - 63.5) / 64
    basis((R)(2 * i - (kBox - 1)) / kBox, b);
    for (int k = 0; k < kQ; ++k) t[kTabP + i * kQ + k] = (double)b[k];
    basis((R)(i - kBox / 2) / (kBox / 2), b);  // point half an integer below it
    for (int k = 0; k < kQ; ++k) t[kTabE + k * kBox + i] = (double)b[k];
  }
  for (int side = 0; side < 2; ++side)  // child nodes in the parent's coordinates
    for (int i = 0; i < kQ; ++i) {
      basis((node[i] + (side ? 1 : -1)) / 2, b);
      for (int k = 0; k < kQ; ++k) t[kTabM + (side * kQ + k) * kQ + i] = (double)b[k];
    }
  // translation downwards, less the value at the child's centre; [side][k][node, centre]
  for (int side = 0; side < 2; ++side) {
    basis(side ? 0.5L : -0.5L, bc);
    for (int i = 0; i <= kQ; ++i) {
      if (i < kQ) basis((node[i] + (side ? 1 : -1)) / 2, b);
      for (int k = 0; k < kQ; ++k)
        t[kTabD + (side * kQ + k) * kQ1 + i] = (double)(i < kQ ? b[k] - bc[k] : bc[k]);
    }
  }
  const int offs[4] = {-3, -2, 2, 3};
  auto kern = [&](int f, int off, R s, R i) {  // (distance between node s and point i)^-(f + 1)
    const R x = 1 / (2 * off + s - i);
    return f ? x * x : x;
  };
  for (int f = 0; f < 2; ++f)
    for (int d = 0; d < 4; ++d) {
      const double c = (double)kern(f, offs[d], 0, 0);
      t[kTabC + f * 4 + d] = c;
      for (int k = 0; k < kQ; ++k) {
        const R at0 = kern(f, offs[d], node[k], 0);
        double* row = &t[kTabK + ((f * 4 + d) * kQ + k) * kQ1];
        for (int i = 0; i < kQ; ++i) row[i] = (double)(kern(f, offs[d], node[k], node[i]) - at0);
        row[kQ] = (double)(at0 - (R)c);
      }
    }
  const R sc = 1 / (4 * (R)kPi2 * (kBox / 2));
  t[kTabSc] = (double)sc;
  t[kTabSc + 1] = (double)(sc * sc);
  for (int f = 0; f < 2; ++f)
    for (int k = 0; k < kQ; ++k)
      for (int i = 0; i < kH; ++i) {
        const R at0 = kern(f, 2, node[k], 0);
        const R a = kern(f, 2, node[k], node[i]) - at0, b2 = kern(f, 2, node[k], -node[i]) - at0;
        t[kTabKS + ((2 * f) * kQ + k) * kH + i] = (double)((a + b2) / 2);
        t[kTabKS + ((2 * f + 1) * kQ + k) * kH + i] = (double)((a - b2) / 2);
      }
  basis(-0.5L, bc);
  for (int i = 0; i <= kQ; ++i) {
    if (i < kQ) basis((node[i] - 1) / 2, b);
    auto at = [&](int k) { return i < kQ ? b[k] - bc[k] : bc[k]; };
    for (int k = 0; k < kH; ++k) {
      t[kTabMS + k * kQ1 + i] = (double)((at(k) + at(kQ - 1 - k)) / 2);
      t[kTabMS + (kH + k) * kQ1 + i] = (double)((at(k) - at(kQ - 1 - k)) / 2);
    }
  }
  for (int l = 0; l < 4 * kBox; ++l) {  // w(l - 256) and its square
    const R w = 1 / ((R)kPi2 * (4 * (l - 2 * kBox) + 2));
    t[kTabW + 2 * l] = (double)w;
    t[kTabW + 2 * l + 1] = (double)(w * w);
  }
  return t;
}

template <int D>
cudaError_t plan_t(lsp_ctx* c) {
  constexpr int NC = Cls<D>::NC;
  FmmPlan& P = c->fmm;
  const int half = c->geo.n / 2;
  const int64_t nr = (int64_t)D * half * half + 1;
  const size_t flag_bytes = (size_t)((nr + 4095) / 4096) * 4096;
  cudaError_t e;
  auto need = [&](DevBuf& b, size_t bytes) { return ensure(c, b, bytes); };
  if (!need(P.tab, sizeof(double) * kTabSize) || !need(P.pos, sizeof(int32_t) * (size_t)nr) ||
      !need(P.rank, flag_bytes) || !need(c->counts, sizeof(int32_t) * (16 + nr / 4096 + 32)))
    return cudaErrorMemoryAllocation;
  static const std::vector<double> t = make_tables();  // constants: once per process
  if ((e = cudaMemcpyAsync(P.tab.p, t.data(), sizeof(double) * kTabSize, cudaMemcpyHostToDevice,
                           c->stream)) != cudaSuccess)
    return e;
  // distinct |p|^2, sorted (the flags live in the buffer of the rank table)
  uint8_t* flag = (uint8_t*)P.rank.p;
  int32_t* counts = (int32_t*)c->counts.p;
  if ((e = launch_zero(c, flag, flag_bytes)) != cudaSuccess) return e;
  const int64_t tuples = D == 2 ? (int64_t)(half + 1) * (half + 1)
                                : (int64_t)(half + 1) * (half + 1) * (half + 1);
  k_fmm_flags<D><<<grid_for(tuples), kThreads, 0, c->stream>>>(half, flag);
  if ((e = launch_compact(c, flag, 0, nr, (int32_t*)P.pos.p, counts + 1, nullptr)) != cudaSuccess)
    return e;
  int32_t ns = 0;
  if ((e = cudaMemcpyAsync(&ns, counts + 1, sizeof ns, cudaMemcpyDeviceToHost, c->stream)) !=
          cudaSuccess ||
      (e = cudaStreamSynchronize(c->stream)) != cudaSuccess)
    return e;
  P.ns = ns;
  int64_t boxes = 0;
  for (int l = 0; l < kFmmLevels; ++l) {
    P.nsb[l] = ((nr - 1) >> (kLog + l)) + 1;
    P.qoff[l] = boxes;
    boxes += P.nsb[l];
  }
  const int64_t words = P.nsb[0] * (kBox / 32) + 1;
  if (!need(P.wgt, sizeof(double) * (size_t)ns * NC) ||
      !need(P.rank, sizeof(uint2) * (size_t)words) ||
      !need(P.q, sizeof(double) * (size_t)boxes * NC * kQ) ||
      !need(P.q0, sizeof(double) * (size_t)boxes * NC))
    return cudaErrorMemoryAllocation;
  const int32_t* pos = (const int32_t*)P.pos.p;
  double* q = (double*)P.q.p;
  const double* tab = (const double*)P.tab.p;
  k_fmm_charges<D><<<grid_for((int64_t)ns * 32), kThreads, 0, c->stream>>>(
      pos, ns, half, (const double*)c->xtab.p, (const double*)c->xtab.p + 5 * (half + 1),
      1.0 / (double)c->geo.N, (double*)P.wgt.p);
  uint2* rank = (uint2*)P.rank.p;
  k_fmm_rank<<<grid_for(words), kThreads, 0, c->stream>>>(pos, ns, words, rank);
  k_fmm_p2m<<<grid_for(P.nsb[0] * NC * kQ), kThreads, 0, c->stream>>>(
      pos, (const double*)P.wgt.p, NC, rank, P.nsb[0], tab, q);
  Levels lv;
  std::copy(P.nsb, P.nsb + kFmmLevels, lv.nsb);
  std::copy(P.qoff, P.qoff + kFmmLevels, lv.qoff);
  int l = 1;
  for (; l < kFmmLevels && P.nsb[l] > 16; ++l)
    k_fmm_m2m<<<grid_for(P.nsb[l] * NC * kQ), kThreads, 0, c->stream>>>(q, lv, l, l + 1, NC, tab);
  if (l < kFmmLevels) k_fmm_m2m<<<1, kThreads, 0, c->stream>>>(q, lv, l, kFmmLevels, NC, tab);
  k_fmm_total<<<grid_for(boxes * NC), kThreads, 0, c->stream>>>(q, boxes * NC, (double*)P.q0.p);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  P.ready = true;
  return cudaSuccess;
}

template <int NC>
cudaError_t build_t(lsp_ctx* c, const int32_t* list, const int32_t* count, int64_t cap) {
  FmmPlan& P = c->fmm;
  const Tree t = fmm_tree(c);
  int32_t* err = (int32_t*)c->counts.p + kErrWord;
  const uint8_t* used = (const uint8_t*)P.used.p;
  double* loc = (double*)P.loc.p;
  const double* q0 = (const double*)P.q0.p;
  const double* tab = (const double*)P.tab.p;
  const int64_t boxes = t.off[t.L + 1];
  cudaError_t e;
  // stage 1: far field at the nodes of the leaf boxes
  int tm = timer_begin(c, "stage1");
  // (a tree of 4 boxes, 3D n = 64: 21.4 us a value per thread, 23.3 a pair per thread)
  const bool few = boxes <= 32;
  e = tuned_launch(c, std::string("stage1/fmm") + std::to_string(NC) + "/w" + work_bucket(boxes),
                   few ? LaunchShape{64, 2} : LaunchShape{kBoxThreads, 32}, kThreads, 0,
                   [&](LaunchShape sh) {
    if (few)  // (one value per thread: no cap)
      k_fmm_m2l<NC><<<(unsigned)((boxes * 2 * NC * kQ1 + sh.threads - 1) / sh.threads), sh.threads,
                      0, c->stream>>>(t, used, tab, (const double*)P.q.p, q0, loc);
    else
      k_fmm_m2l_box<NC><<<(unsigned)std::min<int64_t>(boxes, 152 * (int64_t)sh.per_sm), sh.threads,
                          0, c->stream>>>(t, used, tab, (const double*)P.q.p, q0, loc);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  if (t.L > 0) {
    // the deepest subtrees that still leave two blocks per SM to do (no more than there are shifts)
    int S = 0;
    auto roots = [&](int l) { return std::min<int64_t>(cap, t.off[l + 1] - t.off[l]); };
    while (S < std::min(t.L, kSubLev) && roots(S + 1) >= 2 * 152) ++S;
    const int grid = (int)(t.off[S + 1] - t.off[S]);
    // At most two leaves per SM: a quarter of the columns per block (65 shifts at 2D n = 1024 61 -> 49 us
    // for both translations, n = 256 25.5 -> 21.8, 3D n = 64 25.1 -> 21.4; all 440 leaves of n = 512 with
    // per-point shifts 51.9 -> 54.1).
    if (S == 0 && roots(0) <= 2 * 152)
      k_fmm_l2l<NC, NC / 2><<<dim3(grid, 4), kThreads, 0, c->stream>>>(t, used, tab, loc, S);
    else
      k_fmm_l2l<NC, 2 * NC><<<grid, kThreads, 0, c->stream>>>(t, used, tab, loc, S);
  }
  timer_end(c, tm);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // stage 2: values at the shifts. The count is on the device; its bound min(cap, N) decides how
  // many threads share a shift (the order of the sums depends on nothing else).
  EvalArgs a;
  a.list = list;
  a.count = count;
  a.pos = (const int32_t*)P.pos.p;
  a.wgt = (const double*)P.wgt.p;
  a.rank = (const uint2*)P.rank.p;
  a.tab = tab;
  a.loc = loc;
  a.jlo = t.jlo[0];
  a.nbox = t.off[1];
  a.nsb = P.nsb[0];
  a.g = (double*)c->gvals.p;
  a.cap = cap;
  a.err = err;
  const int64_t bound = std::min<int64_t>(cap, c->geo.N);
  tm = timer_begin(c, "stage2");
  if (bound <= kFmmBlockShifts) {
    k_fmm_eval_block<NC><<<(int)std::max<int64_t>(1, std::min<int64_t>(bound, 152 * 8)), kEvalBlock,
                           0, c->stream>>>(a);
    e = cudaGetLastError();
  } else {
    const int lanes = bound <= kFmmLaneShifts ? 8 : 2;
    e = tuned_launch(c, std::string("stage2/fmm") + std::to_string(NC) + "/lanes" +
                            std::to_string(lanes) + "/w" + work_bucket(bound),
                     {64, 16}, kThreads, 0, [&](LaunchShape sh) {
      const int64_t per = sh.threads / lanes;
      const int64_t b = std::min<int64_t>((bound + per - 1) / per, 152 * (int64_t)sh.per_sm);
      if (lanes == 8)
        k_fmm_eval<NC, 8><<<(int)b, sh.threads, 0, c->stream>>>(a);
      else
        k_fmm_eval<NC, 2><<<(int)b, sh.threads, 0, c->stream>>>(a);
      return cudaGetLastError();
    });
  }
  timer_end(c, tm);
  return e;
}

}  // namespace

cudaError_t fmm_plan(lsp_ctx* c) {
  if (c->fmm.ready) return cudaSuccess;
  return c->geo.d == 2 ? plan_t<2>(c) : plan_t<3>(c);
}

FmmTree fmm_tree(const lsp_ctx* c) {
  const FmmPlan& P = c->fmm;
  FmmTree t;
  const int64_t plo = -c->mrange.hi, phi = -c->mrange.lo;  // integers of the points
  const int64_t lo = std::min<int64_t>(plo, 0);
  const int64_t hi = std::max<int64_t>(phi, (P.nsb[0] << kLog) - 1);
  t.L = 0;
  while (t.L + 2 < kFmmLevels && (hi >> (kLog + t.L + 1)) - (lo >> (kLog + t.L + 1)) > 1) ++t.L;
  t.off[0] = 0;
  for (int l = 0; l < kFmmLevels; ++l) {
    t.jlo[l] = plo >> (kLog + l);
    t.nsb[l] = P.nsb[l];
    t.qoff[l] = P.qoff[l];
    t.off[l + 1] = t.off[l] + (phi >> (kLog + l)) - t.jlo[l] + 1;
  }
  return t;
}

bool fmm_buffers(lsp_ctx* c) {
  const FmmTree t = fmm_tree(c);
  const int64_t boxes = t.off[t.L + 1];
  const int nc = c->geo.d == 2 ? Cls<2>::NC : Cls<3>::NC;
  c->fmm.used_bytes = (size_t)(boxes + 3) / 4 * 4;
  return ensure(c, c->fmm.used, c->fmm.used_bytes) &&
         ensure(c, c->fmm.loc, sizeof(double) * (size_t)boxes * 2 * nc * kRows);
}

cudaError_t launch_fmm_mark(lsp_ctx* c, const int32_t* list, const int32_t* count, int64_t cap) {
  const int tm = timer_begin(c, "fmm_mark");
  k_fmm_mark<<<grid_for(cap), kThreads, 0, c->stream>>>(
      list, count, fmm_tree(c), (uint8_t*)c->fmm.used.p, (int32_t*)c->counts.p + kErrWord);
  timer_end(c, tm);
  return cudaGetLastError();
}

cudaError_t launch_fmm(lsp_ctx* c, const int32_t* list, const int32_t* count, int64_t cap) {
  return c->geo.d == 2 ? build_t<Cls<2>::NC>(c, list, count, cap)
                       : build_t<Cls<3>::NC>(c, list, count, cap);
}

void fmm_free(FmmPlan& P) {
  for (DevBuf* b : {&P.tab, &P.pos, &P.wgt, &P.rank, &P.q, &P.q0, &P.used, &P.loc})
    if (b->p) cudaFree(b->p);
}

}  // namespace lsp
