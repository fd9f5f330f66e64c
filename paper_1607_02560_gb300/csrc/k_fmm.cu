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
// moments depend on n only and are made once per context; 19 200 per box (6900 boxes; 12 000 where
// mirrored nodes share the work, see k_fmm_m2l_box and k_fmm_l2l) for the translations, 970 per
// shift at the end. Fewer nodes or smaller boxes trade these against each other: without the
// mirroring boxes of 64 cost 266e6 + 56e6, of 256 67e6 + 158e6, of 128 133e6 + 90e6.
// Accuracy against extended precision, 2D n = 1024, largest error relative to the largest g of the
// shift: f = 1 1.9e-15 (stages 1.3e-15), f = 2 5e-16 (stages 1e-15); rms 2.6e-16 and 0.9e-16
// (stages 2.4e-16 and 2e-16).
// Measured (both stages, GB300; stage by stage before): 2D n = 1024 per-point shifts 3.68 -> 0.42 ms,
// 65 shifts 0.39 -> 0.06 ms, n = 512 0.49 -> 0.13 ms, n = 256 0.155 -> 0.051 ms, n = 128 0.052 ->
// 0.039 ms, 3D n = 64 0.047 -> 0.033 ms (and two launches fewer for the stage lists).
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

// Device tables of the plan (doubles): P2M [128][20], M2M [2][20][20], M2L [2][4][20][20]
// (f = 1, 2; offsets -3, -2, 2, 3), L2P [20][128], near w [512][2], and for the symmetric pairs (see
// k_fmm_m2l_box and k_fmm_l2l) the half sums and half differences of M2L [2][2][20][10] at offset 2
// and of the interpolation to the lower child [2][10][20].
constexpr int kH = kQ / 2;
constexpr int kTabP = 0, kTabM = kTabP + kBox * kQ, kTabK = kTabM + 2 * kQ * kQ,
              kTabE = kTabK + 8 * kQ * kQ, kTabW = kTabE + kQ * kBox,
              kTabKS = kTabW + 4 * kBox * 2, kTabMS = kTabKS + 4 * kQ * kH,
              kTabSize = kTabMS + 2 * kH * kQ;
static_assert(kTabW % 2 == 0, "16-byte aligned");

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

// Charges of source s (one warp): the tuples with |p|^2 = r, the last component from the others.
template <int D>
__global__ void __launch_bounds__(kThreads) k_fmm_charges(const int32_t* __restrict__ pos, int ns,
                                                          int half, const double* __restrict__ X,
                                                          double inv_n, double* __restrict__ wgt) {
  constexpr int NC = Cls<D>::NC;
  const int P = half + 1, lane = threadIdx.x & 31;
  for (int64_t s = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; s < ns;
       s += ((int64_t)gridDim.x * kThreads) >> 5) {
    const int r = pos[s];
    double acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0.0;
    const int total = D == 2 ? P : P * P;
    for (int e = lane; e < total; e += 32) {
      const int p = D == 2 ? e : e / P, q = D == 2 ? 0 : e - p * P;
      const int rest = r - p * p - q * q;
      if (rest < 0) continue;
      const int z = isqrt_exact(rest);
      if (z * z != rest || z > half) continue;
      if (D == 2) {
        int c = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = a; b < 3; ++b, ++c) acc[c] = fma(X[a * P + p], X[b * P + z], acc[c]);
      } else {
        int c = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = a; b < 3; ++b)
#pragma unroll
            for (int g = b; g < 3; ++g, ++c)
              acc[c < NC ? c : 0] =
                  fma(X[a * P + p] * X[b * P + q], X[g * P + z], acc[c < NC ? c : 0]);
      }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
      if (lane == 0) wgt[s * NC + c] = acc[c] * inv_n;
    }
  }
}

// start[j] = first source at or beyond integer 128 j, j = 0..nbox.
__global__ void __launch_bounds__(kThreads) k_fmm_start(const int32_t* __restrict__ pos, int ns,
                                                        int64_t nbox, int32_t* __restrict__ start) {
  for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j <= nbox;
       j += (int64_t)gridDim.x * kThreads) {
    int lo = 0, hi = ns;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (pos[mid] < j * kBox)
        lo = mid + 1;
      else
        hi = mid;
    }
    start[j] = lo;
  }
}

// Moments of the leaf boxes, q[box][c][k] = sum over the box' sources of N_c(r) L_k(r).
__global__ void __launch_bounds__(kThreads) k_fmm_p2m(const int32_t* __restrict__ pos,
                                                      const double* __restrict__ wgt, int nc,
                                                      const int32_t* __restrict__ start,
                                                      int64_t nbox, const double* __restrict__ tab,
                                                      double* __restrict__ q) {
  const int64_t total = nbox * nc * kQ;
  for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * kThreads) {
    const int k = (int)(e % kQ), c = (int)(e / kQ % nc);
    const int64_t b = e / kQ / nc;
    double acc = 0.0;
    for (int s = start[b]; s < start[b + 1]; ++s)
      acc = fma(wgt[(int64_t)s * nc + c], tab[kTabP + (pos[s] & (kBox - 1)) * kQ + k], acc);
    q[e] = acc;
  }
}

// Moments of the parent boxes of levels l0 .. l1 - 1 from their children (box 2 b + side). The
// lowest levels take a launch each; from where one block covers a level, one block does the rest.
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

// Node values from the boxes two or three apart (children of the parent's neighbours; offsets
// -2, 2, 3 of even boxes, -3, -2, 2 of odd ones: indices 0..3 = -3, -2, 2, 3), every level at once:
// they need only the moments. One thread per value, tables and moments through L1. FP64 pipe.
// Measured with the translation downwards (before: a block per box, tables in shared memory): 2D
// n = 1024 233 -> 216 us, n = 512 59 -> 52 us, n = 32 17.3 -> 15.2 us, 3D n = 64 29.6 -> 25.1 us.
template <int NC>
__global__ void __launch_bounds__(kThreads) k_fmm_m2l(const __grid_constant__ Tree t,
                                                             const uint8_t* __restrict__ used,
                                                             const double* __restrict__ tab,
                                                             const double* __restrict__ q,
                                                             double* __restrict__ loc) {
  constexpr int FC = 2 * NC, OUT = FC * kQ;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, u = e / OUT;
  if (u >= t.off[t.L + 1] || !used[u]) return;
  const int o = (int)(e - u * OUT), i = o / FC, fc = o - i * FC, c = fc >> 1, f = fc & 1;
  int l = 0;
  while (u >= t.off[l + 1]) ++l;
  const int64_t j = t.jlo[l] + (u - t.off[l]);
  double acc = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int di = d + 1 - (int)(j & 1);
    const int64_t x = j + (di < 2 ? di - 3 : di);
    if (x < 0 || x >= t.nsb[l]) continue;
    const double* K = tab + kTabK + ((f * 4 + di) * kQ) * kQ + i;
    const double* qq = q + (t.qoff[l] + x) * (NC * kQ) + c * kQ;
#pragma unroll
    for (int k = 0; k < kQ; ++k) acc = fma(__ldg(K + k * kQ), __ldg(qq + k), acc);
  }
  const double sc = (1.0 / (4.0 * kPi2)) * (1.0 / (double)((int64_t)(kBox / 2) << l));
  loc[e] = acc * (f ? sc * sc : sc);
}

// The same, a block per box and a thread per pair of mirrored nodes (i, 19 - i). With R the moments
// of the box at offset 2 and L those at -2 in reverse order, K_-2[k][i] = -+K_2[19 - k][19 - i] (f = 1,
// 2) gives
//   out[i] + out[19 - i] = sum_k (K_2[k][i] + K_2[k][19 - i]) (R -+ L)[k],
//   out[i] - out[19 - i] = sum_k (K_2[k][i] - K_2[k][19 - i]) (R +- L)[k],
// 80 instead of 120 multiply-adds a pair with the third offset. Measured with the translation
// downwards: 2D n = 1024 208 -> 175 us, n = 512 53.7 -> 50.0 us, n = 128 20.5 -> 18.7 us.
template <int NC>
__global__ void __launch_bounds__(NC * kQ) k_fmm_m2l_box(const __grid_constant__ Tree t,
                                                         const uint8_t* __restrict__ used,
                                                         const double* __restrict__ tab,
                                                         const double* __restrict__ q,
                                                         double* __restrict__ loc) {
  constexpr int FC = 2 * NC, OUT = FC * kQ;
  __shared__ double sa[2][NC][kQ], s3[NC][kQ];  // R + L, R - L; the moments at offset 3 or -3
  const int64_t u = blockIdx.x;
  if (!used[u]) return;
  int l = 0;
  while (u >= t.off[l + 1]) ++l;
  const int64_t j = t.jlo[l] + (u - t.off[l]);
  const int odd = (int)(j & 1);
  {
    const int c = threadIdx.x / kQ, k = threadIdx.x % kQ;
    auto moment = [&](int64_t x, int kk) {
      return x >= 0 && x < t.nsb[l] ? __ldg(q + (t.qoff[l] + x) * (NC * kQ) + c * kQ + kk) : 0.0;
    };
    const double r = moment(j + 2, k), m = moment(j - 2, kQ - 1 - k);
    sa[0][c][k] = r + m;
    sa[1][c][k] = r - m;
    s3[c][k] = moment(odd ? j - 3 : j + 3, k);
  }
  __syncthreads();
  const int i = threadIdx.x / FC, fc = threadIdx.x - i * FC, c = fc >> 1, f = fc & 1;
  const double* KS = tab + kTabKS + 2 * f * kQ * kH + i;
  const double* K3 = tab + kTabK + ((f * 4 + (odd ? 0 : 3)) * kQ) * kQ + i;
  const double *ps = sa[1 - f][c], *pd = sa[f][c], *p3 = s3[c];
  double sum = 0.0, dif = 0.0, lo = 0.0, hi = 0.0;
#pragma unroll
  for (int k = 0; k < kQ; ++k) {
    sum = fma(__ldg(KS + k * kH), ps[k], sum);
    dif = fma(__ldg(KS + (kQ + k) * kH), pd[k], dif);
    lo = fma(__ldg(K3 + k * kQ), p3[k], lo);
    hi = fma(__ldg(K3 + k * kQ + kQ - 1 - 2 * i), p3[k], hi);
  }
  const double sc1 = (1.0 / (4.0 * kPi2)) * (1.0 / (double)((int64_t)(kBox / 2) << l));
  const double sc = f ? sc1 * sc1 : sc1;
  loc[u * OUT + i * FC + fc] = (lo + (sum + dif)) * sc;
  loc[u * OUT + (kQ - 1 - i) * FC + fc] = (hi + (sum - dif)) * sc;
}

// Node values of the leaves: from the top, child = own + interpolation of the parent's. A block
// follows the path to one box of level S <= 3, then the boxes below it: S = 3 repeats the least of
// the upper levels' work (2D n = 1024: 50e6 FP64 instructions, S = 0 183e6), smaller S spreads
// a small tree over more SMs (2D n = 128, 55 leaves: both passes 40 -> 25 us).
// FS of the 2 NC columns (class, f) per block: they are independent of each other.
template <int NC, int FS>
__global__ void __launch_bounds__(kThreads) k_fmm_l2l(const __grid_constant__ Tree t,
                                                      const uint8_t* __restrict__ used,
                                                      const double* __restrict__ tab,
                                                      double* __restrict__ loc, int S) {
  constexpr int FC = 2 * NC, ALL = FC * kQ, OUT = FS * kQ;
  const int f0 = blockIdx.y * FS;
  auto at = [&](int64_t u, int o) {  // place of value o of this block's columns of box u
    return u * ALL + o / FS * FC + f0 + o % FS;
  };
  __shared__ double sM[2 * kQ * kQ], sS[2 * kH * kQ];
  __shared__ double buf[2][(1 << (kSubLev - 1)) * OUT];  // levels S - 1.. 1 at most 4 boxes
  const int64_t root = blockIdx.x;  // box of level S
  if (t.L == 0 || !used[t.off[S] + root]) return;
  for (int e = threadIdx.x; e < 2 * kQ * kQ; e += kThreads) sM[e] = tab[kTabM + e];
  for (int e = threadIdx.x; e < 2 * kH * kQ; e += kThreads) sS[e] = tab[kTabMS + e];
  const int64_t jr = t.jlo[S] + root;
  // from the parent's node values src to those of a child on the given side
  auto down = [&](const double* src, int side, int o) -> double {
    const int i = o / FS, fc = o - i * FS;
    const double* M = sM + side * kQ * kQ + i;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < kQ; ++k) acc = fma(M[k * kQ], src[k * FS + fc], acc);
    return acc;
  };
  int cur = 0;
  {
    const int64_t u = t.off[t.L] + (jr >> (t.L - S)) - t.jlo[t.L];
    for (int o = threadIdx.x; o < OUT; o += kThreads) buf[0][o] = loc[at(u, o)];
  }
  __syncthreads();
  for (int l = t.L - 1; l >= S; --l, cur ^= 1) {
    const int64_t j = jr >> (l - S), u = t.off[l] + j - t.jlo[l];
    for (int o = threadIdx.x; o < OUT; o += kThreads) {
      const double v = loc[at(u, o)] + down(buf[cur], (int)(j & 1), o);
      if (l == 0)
        loc[at(u, o)] = v;
      else
        buf[cur ^ 1][o] = v;
    }
    __syncthreads();
  }
  if constexpr (FS < FC) {
    for (int l = S - 1; l >= 0; --l, cur ^= 1) {
      const int nb = 1 << (S - l);  // boxes of this level under the root
      for (int e = threadIdx.x; e < nb * OUT; e += kThreads) {
        const int b = e / OUT, o = e - b * OUT;
        const int64_t x = (jr << (S - l)) + b - t.jlo[l], u = t.off[l] + x;
        if (x < 0 || u >= t.off[l + 1] || !used[u]) continue;
        const double v = loc[at(u, o)] + down(buf[cur] + (b >> 1) * OUT, b & 1, o);
        if (l == 0)
          loc[at(u, o)] = v;
        else
          buf[cur ^ 1][b * OUT + o] = v;
      }
      __syncthreads();
    }
    return;
  }
  // All columns: both children of a parent together. With e, o the sums and differences of its values
  // at mirrored nodes, node i of the lower child is E + O and node 19 - i of the upper one E - O,
  // E = sum_k<10 Ms[k][i] e[k], O = sum Md[k][i] o[k]: half the multiply-adds for one more barrier a
  // level (2D n = 1024, both translations 216 -> 208 us; with few subtrees the barrier costs more:
  // 3D n = 64 21.4 -> 23.5 us).
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
    for (int e = threadIdx.x; e < np * OUT; e += kThreads) {
      const int b = e / OUT, o = e - b * OUT, i = o / FS, fc = o - i * FS;
      const int64_t x = (jr << (S - l)) + 2 * b - t.jlo[l], u = t.off[l] + x;  // the lower child
      const bool lower = x >= 0 && u < t.off[l + 1] && used[u];
      const bool upper = x + 1 >= 0 && u + 1 < t.off[l + 1] && used[u + 1];
      if (!lower && !upper) continue;
      const double* src = par + b * OUT + fc;
      double E = 0.0, O = 0.0;
#pragma unroll
      for (int k = 0; k < kH; ++k) {
        E = fma(sS[k * kQ + i], src[k * FS], E);
        O = fma(sS[(kH + k) * kQ + i], src[(kQ - 1 - k) * FS], O);
      }
      const int om = (kQ - 1 - i) * FS + fc;  // the mirrored node
      if (lower) {
        const double v = loc[at(u, o)] + (E + O);
        if (l == 0)
          loc[at(u, o)] = v;
        else
          buf[cur ^ 1][2 * b * OUT + o] = v;
      }
      if (upper) {
        const double v = loc[at(u + 1, om)] + (E - O);
        if (l == 0)
          loc[at(u + 1, om)] = v;
        else
          buf[cur ^ 1][(2 * b + 1) * OUT + om] = v;
      }
    }
    __syncthreads();
  }
}

struct EvalArgs {
  const int32_t* list;
  const int32_t* count;
  const int32_t* pos;
  const double* wgt;
  const int32_t* start;
  const double* tab;
  const double* loc;
  int64_t jlo, nbox, nsb;
  double* g;
  int64_t cap;
  int32_t* err;
};

// The sums of one shift over this lane's share: nodes lane, lane + LANES, ... of the far part and
// every LANES-th near source.
template <int NC>
__device__ __forceinline__ void eval_part(const EvalArgs& a, int64_t m, int lane, int lanes,
                                          const double* sE, const double2* sW,
                                          double (&acc)[2 * NC]) {
  const int64_t x = -m, j = x >> kLog, b = checked(j - a.jlo, a.nbox, a.err);
  const int tp = (int)(x & (kBox - 1));
  const double* lo = a.loc + b * (2 * NC * kQ);
#pragma unroll
  for (int c = 0; c < 2 * NC; ++c) acc[c] = 0.0;
  for (int i = lane; i < kQ; i += lanes) {
    const double e = sE[i * kBox + tp];
    const double2* v = reinterpret_cast<const double2*>(lo + i * 2 * NC);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const double2 q = __ldg(v + c);
      acc[2 * c] = fma(q.x, e, acc[2 * c]);
      acc[2 * c + 1] = fma(q.y, e, acc[2 * c + 1]);
    }
  }
  auto clampb = [&](int64_t k) { return k < 0 ? (int64_t)0 : (k > a.nsb ? a.nsb : k); };
  const int s0 = __ldg(a.start + clampb(j - 1)), s1 = __ldg(a.start + clampb(j + 2));
  for (int s = s0 + lane; s < s1; s += lanes) {
    const double2 w = sW[(int)(__ldg(a.pos + s) + m) + 2 * kBox];
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

// g values of every shift, LANES threads per shift: 2 for long lists (2D n = 1024: 1, 2, 4, 8 lanes
// 250, 243, 252, 327 us; one lane leaves too few warps, more repeat the far part's loads and the
// reduction), 8 for short ones (2D n = 256: 68, 38, 30, 30 us; n = 128: 75, 42, 28, 20 us). The
// tables are read through L1 (28 KiB).
template <int NC, int LANES>
__global__ void __launch_bounds__(kThreads) k_fmm_eval(EvalArgs a) {
  const double* sE = a.tab + kTabE;
  const double2* sW = reinterpret_cast<const double2*>(a.tab + kTabW);
  const int64_t cnt = *a.count;
  const int lane = threadIdx.x % LANES;
  const int64_t step = (int64_t)gridDim.x * (blockDim.x / LANES);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x / LANES) + threadIdx.x / LANES;
       __any_sync(0xffffffffu, i < cnt); i += step) {
    double acc[2 * NC];
    const bool live = i < cnt;
    eval_part<NC>(a, __ldg(a.list + (live ? i : 0)), lane, LANES, sE, sW, acc);
#pragma unroll
    for (int c = 0; c < 2 * NC; ++c) {
#pragma unroll
      for (int o = LANES / 2; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
      if (live && lane == 0) a.g[(int64_t)c * a.cap + i] = acc[c];
    }
  }
}

// Few shifts: a block of 128 threads (all four FP64 quarters of an SM) per shift. The 128
// partial sums of each value are added by eight lanes, 16 each, then across them.
constexpr int kEvalBlock = 128;
template <int NC>
__global__ void __launch_bounds__(kEvalBlock) k_fmm_eval_block(EvalArgs a) {
  constexpr int FC = 2 * NC;
  __shared__ double part[FC][kEvalBlock + 1];
  const double2* sW = reinterpret_cast<const double2*>(a.tab + kTabW);  // few values: read in L1
  const int64_t cnt = *a.count;
  for (int64_t i = blockIdx.x; i < cnt; i += gridDim.x) {
    double acc[FC];
    eval_part<NC>(a, __ldg(a.list + i), threadIdx.x, kEvalBlock, a.tab + kTabE, sW, acc);
#pragma unroll
    for (int c = 0; c < FC; ++c) part[c][threadIdx.x] = acc[c];
    __syncthreads();
    const int sub = threadIdx.x & 7;
    for (int c = threadIdx.x >> 3; c < (FC + 15) / 16 * 16; c += kEvalBlock / 8) {
      double s = 0.0;
      if (c < FC)
        for (int k = sub; k < kEvalBlock; k += 8) s += part[c][k];
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (c < FC && sub == 0) a.g[(int64_t)c * a.cap + i] = s;
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
  R b[kQ];
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
  const int offs[4] = {-3, -2, 2, 3};
  for (int d = 0; d < 4; ++d)
    for (int k = 0; k < kQ; ++k)
      for (int i = 0; i < kQ; ++i) {
        const R x = 1 / (2 * offs[d] + node[k] - node[i]);
        t[kTabK + (d * kQ + k) * kQ + i] = (double)x;
        t[kTabK + ((4 + d) * kQ + k) * kQ + i] = (double)(x * x);
      }
  for (int f = 0; f < 2; ++f)
    for (int k = 0; k < kQ; ++k)
      for (int i = 0; i < kH; ++i) {
        const R x = 1 / (4 + node[k] - node[i]), y = 1 / (4 + node[k] + node[i]);
        const R a = f ? x * x : x, b2 = f ? y * y : y;
        t[kTabKS + ((2 * f) * kQ + k) * kH + i] = (double)((a + b2) / 2);
        t[kTabKS + ((2 * f + 1) * kQ + k) * kH + i] = (double)((a - b2) / 2);
      }
  for (int i = 0; i < kQ; ++i) {
    basis((node[i] - 1) / 2, b);
    for (int k = 0; k < kH; ++k) {
      t[kTabMS + k * kQ + i] = (double)((b[k] + b[kQ - 1 - k]) / 2);
      t[kTabMS + (kH + k) * kQ + i] = (double)((b[k] - b[kQ - 1 - k]) / 2);
    }
  }
  for (int l = 0; l < 4 * kBox; ++l) {  // w(l - 256) and its square, as the stages' table
    const double w = 1.0 / (kPi2 * (double)(4 * (l - 2 * kBox) + 2));
    t[kTabW + 2 * l] = w;
    t[kTabW + 2 * l + 1] = w * w;
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
      !need(P.start, flag_bytes) || !need(c->counts, sizeof(int32_t) * (16 + nr / 4096 + 32)))
    return cudaErrorMemoryAllocation;
  static const std::vector<double> t = make_tables();  // constants: once per process
  if ((e = cudaMemcpyAsync(P.tab.p, t.data(), sizeof(double) * kTabSize, cudaMemcpyHostToDevice,
                           c->stream)) != cudaSuccess)
    return e;
  // distinct |p|^2, sorted (the flags live in the buffer of the leaf lists)
  uint8_t* flag = (uint8_t*)P.start.p;
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
  if (!need(P.wgt, sizeof(double) * (size_t)ns * NC) ||
      !need(P.start, sizeof(int32_t) * (size_t)(P.nsb[0] + 1)) ||
      !need(P.q, sizeof(double) * (size_t)boxes * NC * kQ))
    return cudaErrorMemoryAllocation;
  const int32_t* pos = (const int32_t*)P.pos.p;
  double* q = (double*)P.q.p;
  const double* tab = (const double*)P.tab.p;
  k_fmm_charges<D><<<grid_for((int64_t)ns * 32), kThreads, 0, c->stream>>>(
      pos, ns, half, (const double*)c->xtab.p, 1.0 / (double)c->geo.N, (double*)P.wgt.p);
  k_fmm_start<<<grid_for(P.nsb[0] + 1), kThreads, 0, c->stream>>>(pos, ns, P.nsb[0],
                                                                  (int32_t*)P.start.p);
  k_fmm_p2m<<<grid_for(P.nsb[0] * NC * kQ), kThreads, 0, c->stream>>>(
      pos, (const double*)P.wgt.p, NC, (const int32_t*)P.start.p, P.nsb[0], tab, q);
  Levels lv;
  std::copy(P.nsb, P.nsb + kFmmLevels, lv.nsb);
  std::copy(P.qoff, P.qoff + kFmmLevels, lv.qoff);
  int l = 1;
  for (; l < kFmmLevels && P.nsb[l] > 16; ++l)
    k_fmm_m2m<<<grid_for(P.nsb[l] * NC * kQ), kThreads, 0, c->stream>>>(q, lv, l, l + 1, NC, tab);
  if (l < kFmmLevels) k_fmm_m2m<<<1, kThreads, 0, c->stream>>>(q, lv, l, kFmmLevels, NC, tab);
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
  const double* tab = (const double*)P.tab.p;
  const int64_t boxes = t.off[t.L + 1];
  cudaError_t e;
  // stage 1: far field at the nodes of the leaf boxes
  int tm = timer_begin(c, "stage1");
  // (a tree of 4 boxes, 3D n = 64: 21.4 us a value per thread, 23.3 a pair per thread)
  const bool few = boxes <= 32;
  e = tuned_launch(c, std::string("stage1/fmm") + std::to_string(NC) + "/w" + work_bucket(boxes),
                   {64, 2}, kThreads, 0, [&](LaunchShape sh) {
    if (few)  // (one value per thread: no cap)
      k_fmm_m2l<NC><<<(unsigned)((boxes * 2 * NC * kQ + sh.threads - 1) / sh.threads), sh.threads,
                      0, c->stream>>>(t, used, tab, (const double*)P.q.p, loc);
    else
      k_fmm_m2l_box<NC><<<(unsigned)boxes, NC * kQ, 0, c->stream>>>(t, used, tab,
                                                                    (const double*)P.q.p, loc);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  if (t.L > 0) {
    // the deepest subtrees that still leave two blocks per SM
    int S = 0;
    while (S < std::min(t.L, kSubLev) && t.off[S + 2] - t.off[S + 1] >= 2 * 152) ++S;
    // At most two subtrees per SM to do (no more than there are shifts): a quarter of the columns
    // per block (65 shifts at 2D n = 1024 61 -> 49 us for both translations, n = 256 25.5 -> 21.8,
    // 3D n = 64 25.1 -> 21.4; all 440 subtrees of n = 512 with per-point shifts 51.9 -> 54.1).
    const int roots = (int)(t.off[S + 1] - t.off[S]);
    if (std::min<int64_t>(cap, roots) <= 2 * 152)
      k_fmm_l2l<NC, NC / 2><<<dim3(roots, 4), kThreads, 0, c->stream>>>(t, used, tab, loc, S);
    else
      k_fmm_l2l<NC, 2 * NC><<<roots, kThreads, 0, c->stream>>>(t, used, tab, loc, S);
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
  a.start = (const int32_t*)P.start.p;
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
         ensure(c, c->fmm.loc, sizeof(double) * (size_t)boxes * 2 * nc * kQ);
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
  for (DevBuf* b : {&P.tab, &P.pos, &P.wgt, &P.start, &P.q, &P.used, &P.loc})
    if (b->p) cudaFree(b->p);
}

}  // namespace lsp
