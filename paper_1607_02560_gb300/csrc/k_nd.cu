// Numeric phases of the nested dissection of P (Sec. 3, Eq. QC; Fig. nd; Table cost), see
// nd.h for the tree and the front layout:
//  - assembly: a front = its children's Schur complements (extend-add through the ring maps)
//    plus P's entries listed for it;
//  - partial inversion of each front on its eliminated set E with row pivoting inside E
//    (Gauss-Jordan sweep): in shared memory for small fronts, else in blocked steps (the panels
//    here, the steps and their rank-kNdStep update on the tensor cores in k_nd_tc.cu);
//  - the solve: one matrix-vector product per front going up the tree, one coming down.
// Every reduction runs in a fixed order, so a factorisation and a solve are deterministic.
#include <math.h>
#include <stdio.h>

#include "nd.h"
#include "recip.cuh"

namespace lsp {
namespace {

constexpr int NP = kNdPanel;

__global__ void k_nd_extend(double* __restrict__ F, const double* __restrict__ Fc,
                            const int32_t* __restrict__ inv, int count, int f, int nchild,
                            int fc, int sc) {
  const int64_t ff = (int64_t)f * f, total = (int64_t)count * ff;
  const int64_t fcc = (int64_t)fc * fc;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = idx / ff;
    const int rem = (int)(idx - p * ff);
    const int i = rem / f, j = rem - i * f;
    const int32_t* iv = inv + p * f * 2;
    double acc = 0.0;
    for (int c = 0; c < nchild; ++c) {
      const int ai = iv[i * 2 + c], aj = iv[j * 2 + c];
      if (ai >= 0 && aj >= 0) {
        const int64_t child = nchild == 1 ? p : 2 * p + c;
        acc += Fc[child * fcc + (int64_t)(sc + ai) * fc + sc + aj];
      }
    }
    F[idx] = acc;
  }
}

__global__ void k_nd_scatter(double* __restrict__ F, const double* __restrict__ rows,
                             const int32_t* __restrict__ dst, const int32_t* __restrict__ src,
                             int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    F[dst[e]] += rows[src[e]];
}

// argmax of |value| over a warp with ties to the smaller index
__device__ __forceinline__ void warp_argmax_f(float& best, int& bi) {
  for (int off = 16; off > 0; off >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, off);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
    if (ob > best || (ob == best && oi < bi)) {
      best = ob;
      bi = oi;
    }
  }
}

// Partial inversion of one front (f <= kNdSmallFront) in shared memory, one pivot at a time.
// Pivot k: the row of largest |F[i][k]| (by its upper 32 bits) among the rows k..s-1 still
// unpivoted, exchanged with row k; then
//   F[k][k] <- 1/F[k][k], F[k][j] <- F[k][j]/F[k][k], F[i][k] <- -F[i][k]/F[k][k],
//   F[i][j] <- F[i][j] - F[i][k] F[k][j]/F[k][k]   (i, j != k).
// A warp updates whole rows, NJ = ceil(f / 32) entries a lane, with its part of the pivot row in
// registers; the exchange is folded into the update. Rows whose multiplier is zero stay as they
// are: in a leaf, whose rows have 9 or 27 entries, a third of them on average.
// What bounds it: the FP64 pipe in the leaves (n = 512: 4096 fronts of 81 rows, 49 pivots) and its
// latency elsewhere. Measured: the leaves of n = 512 3.90 -> 2.84 ms (before: every row and entry
// updated, FP64 comparisons and a division per pivot, the exchange as a pass of its own).
template <int NJ>
__global__ void __launch_bounds__(512) k_nd_sweep_small(double* __restrict__ fronts, int f, int s,
                                                        int32_t* __restrict__ perm,
                                                        int32_t* __restrict__ err) {
  extern __shared__ double sm[];
  double* F = sm;
  double* colk = F + f * f;  // column k (of the row that takes each position)
  double* rowk = colk + f;   // the scaled pivot row
  double* rowo = rowk + f;   // row k before the exchange
  __shared__ int sperm[kNdSmallFront];
  __shared__ int piv, bad;
  __shared__ double spiv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = blockDim.x;
  double* G = fronts + (int64_t)blockIdx.x * f * f;
  for (int e = tid; e < f * f; e += nt) F[e] = G[e];
  for (int e = tid; e < s; e += nt) sperm[e] = e;
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int k = 0; k < s; ++k) {
    if (warp == 0) {
      unsigned key = 0;
      int bi = k;
      for (int i = k + lane; i < s; i += 32) {
        const unsigned a = ((unsigned)__double2hiint(F[i * f + k]) & 0x7fffffffu) + 1u;
        if (a > key) {
          key = a;
          bi = i;
        }
      }
      const unsigned top = __reduce_max_sync(0xffffffffu, key);
      const int p = (int)__reduce_min_sync(0xffffffffu, key == top ? (unsigned)bi : 0xffffffffu);
      if (lane == 0) {
        const double x = F[p * f + k];
        if (x == 0.0 || top > 0x7ff00000u) {  // zero, Inf or NaN
          bad = 1;
          atomicOr(err, 1);
        }
        piv = p;
        spiv = recip_f64(x);
        const int t = sperm[k];
        sperm[k] = sperm[p];
        sperm[p] = t;
      }
    }
    __syncthreads();
    if (bad) break;
    const int p = piv;
    const double dinv = spiv;
    if (tid < f) {
      rowk[tid] = F[p * f + tid] * dinv;
      rowo[tid] = F[k * f + tid];
      colk[tid] = F[(tid == p ? k : tid) * f + k];
    }
    __syncthreads();
    double rk[NJ];
#pragma unroll
    for (int c = 0; c < NJ; ++c) {
      const int j = lane + 32 * c;
      rk[c] = j < f ? (j == k ? dinv : rowk[j]) : 0.0;
    }
    for (int i = warp; i < f; i += nt / 32) {
      double* Fi = F + i * f;
      const double* Fo = i == p ? rowo : Fi;
      const double ci = i == k ? -1.0 : colk[i];
      if (ci == 0.0 && i != p) continue;
#pragma unroll
      for (int c = 0; c < NJ; ++c) {
        const int j = lane + 32 * c;
        if (j < f) Fi[j] = fma(-ci, rk[c], j == k || i == k ? 0.0 : Fo[j]);
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < f * f; e += nt) G[e] = F[e];
  for (int e = tid; e < s; e += nt) perm[(int64_t)blockIdx.x * s + e] = sperm[e];
}

// ---- blocked partial inversion (k_nd_tc.cu): panels of the sub-steps K = [k, k + nb) of a step
// with the columns [k0, k0 + sb) ----
// swaps layout per front: [0] = number of entries q, then the positions that get another row after
// the sub-step, in the order of their rows in xrow; the first nb are the pivot rows.
constexpr int kSwapInts = kNdSwapInts, SB = kNdStep;

// FP32 value of x for ranking pivot candidates, from the high word of the IEEE double: sign,
// exponent rebased from 1023 to 127, the top 20 fraction bits (relative error < 2^-20);
// magnitudes below the FP32 normal range give 0, above it infinity. Integer operations only.
__device__ __forceinline__ float rank_f32(double x) {
  const int hi = __double2hiint(x);
  const int e = ((hi >> 20) & 0x7ff) - (1023 - 127);
  const unsigned sign = (unsigned)hi & 0x80000000u;
  if (e <= 0) return __uint_as_float(sign);
  if (e >= 255) return __uint_as_float(sign | 0x7f800000u);
  return __uint_as_float(sign | ((unsigned)e << 23) | (((unsigned)hi & 0xfffffu) << 3));
}

// Common end (after the pivot rows sel[0..nb) are known, block-synchronised): row exchanges, the
// exchanged rows' columns of the step, the FP64 pivot-block inverse.
__device__ __forceinline__ void panel_tail(const double* F, int f, int s, int k,
                                           int nb, int k0, int sb, int64_t fid, const int* sel,
                                           int32_t* perm, int32_t* cur,
                                           double* xrow, double* pinv,
                                           int32_t* swaps, int32_t* err) {
  constexpr int NT = 256;
  __shared__ int nq;
  __shared__ int dstp[2 * NP], srcp[2 * NP];
  __shared__ double A[2][NP][NP + 1], trow[2][NP];
  __shared__ int piv_row[NP], row_piv[NP];  // p_j, and the j of a row
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gr = tid / NP, gc = tid % NP;  // 256 threads = 16 x 16
  // the pivot block and the pivot rows' columns of the step: loads that need only the choice
  double* xr = xrow + fid * (2 * NP * SB);
  double keep[NP * SB / NT], moved[NP * SB / NT];
  A[0][gr][gc] = gr < nb && gc < nb ? F[(int64_t)(k + sel[gr]) * f + k + gc] : 0.0;
#pragma unroll
  for (int u = 0; u < NP * SB / NT; ++u) {
    const int e = tid + u * NT, a = e / SB, c = e % SB;
    keep[u] = a < nb && c < sb ? F[(int64_t)(k + sel[a]) * f + k0 + c] : 0.0;
  }
  // row exchanges (the last warp): position k + j takes the row chosen j-th; the rows of K that
  // were not chosen move, in increasing position order, to the positions the chosen rows left
  // outside K (taken in choice order)
  if (warp == NT / 32 - 1) {
    const bool act = lane < nb;
    const int ps = act ? k + sel[lane] : 0;
    const bool inK = act && ps < k + nb;
    const unsigned selK = __reduce_or_sync(0xffffffffu, inK ? 1u << (ps - k) : 0u);
    const unsigned full = nb >= 32 ? 0xffffffffu : (1u << nb) - 1u;
    const unsigned displaced = ~selK & full;  // K positions whose rows were not chosen
    const unsigned outb = __ballot_sync(0xffffffffu, act && !inK);
    const int rank = __popc(outb & ((1u << lane) - 1u));  // among the chosen rows outside K
    int dpos = -1;
    if (act && !inK) {  // the rank-th displaced position of K
      unsigned mk = displaced;
      for (int t = 0; t < rank; ++t) mk &= mk - 1u;
      dpos = k + __ffs(mk) - 1;
    }
    const int nout = __popc(outb);
    int32_t* pf = perm + fid * s;
    int32_t* cf = cur + fid * s;
    int32_t* sw = swaps + fid * kSwapInts;
    const int old_sel = act ? pf[ps] : 0, cur_sel = act ? cf[ps] : 0;
    const int old_dis = dpos >= 0 ? pf[dpos] : 0, cur_dis = dpos >= 0 ? cf[dpos] : 0;
    __syncwarp();
    if (act) {
      dstp[lane] = k + lane;
      srcp[lane] = ps;
      pf[k + lane] = old_sel;
      cf[k + lane] = cur_sel;
    }
    if (dpos >= 0) {
      dstp[nb + rank] = ps;
      srcp[nb + rank] = dpos;
      pf[ps] = old_dis;
      cf[ps] = cur_dis;
    }
    __syncwarp();
    const int qq = nb + nout;
    if (lane == 0) {
      nq = qq;
      sw[0] = qq;
    }
    for (int a = lane; a < qq; a += 32) sw[1 + a] = dstp[a];
  }
  __syncthreads();
  // the displaced rows' columns, stored after the inversion, which covers the latency
  const int q = nq;
#pragma unroll
  for (int u = 0; u < NP * SB / NT; ++u) {
    const int e = tid + u * NT, a = nb + e / SB, c = e % SB;
    moved[u] = a < q && c < sb ? F[(int64_t)srcp[a] * f + k0 + c] : 0.0;
  }
  // Inverse of the pivot block A (FP64): Gauss-Jordan in place, one element per thread, no row
  // exchanges: pivot j is taken in the unpivoted row p_j of largest |a_pj,j| (by the upper 32 bits),
  // row p_j is scaled by one reciprocal, column j is eliminated from the other rows. Row p_j,
  // column c of the result is element (j, p_c) of A^-1. Warp 0 prepares pivot j + 1 (column, choice,
  // reciprocal, scaled row) while the others eliminate pivot j: one barrier a pivot.
  bool open = lane < nb;  // warp 0: the lane's row has not been a pivot row
  auto choose = [&](int j, double x) {  // x: column j of row lane % 16; the pivot's reciprocal
    const unsigned key = open ? ((unsigned)__double2hiint(x) & 0x7fffffffu) + 1u : 0u;
    const unsigned top = __reduce_max_sync(0xffffffffu, key);
    const int p = __ffs(__ballot_sync(0xffffffffu, key == top)) - 1;
    const double xp = __shfl_sync(0xffffffffu, x, p);
    if (lane == p) {
      open = false;
      if (x == 0.0 || top > 0x7ff00000u) atomicOr(err, 4);  // zero, Inf or NaN
      piv_row[j] = p;
      row_piv[p] = j;
    }
    return make_double2(recip_f64(xp), __hiloint2double(0, p));
  };
  const int lr = lane & (NP - 1);
  if (warp == 0) {
    const double2 d = choose(0, A[0][lr][0]);
    const int p = __double2loint(d.y);
    if (lane < NP) trow[0][lane] = lane == 0 ? d.x : A[0][p][lane] * d.x;
  }
  __syncthreads();
  for (int j = 0; j < nb; ++j) {
    const double(*Aj)[NP + 1] = A[j & 1];
    double(*An)[NP + 1] = A[~j & 1];
    const double* tj = trow[j & 1];
    const int p = piv_row[j];
    if (warp == 0 && j + 1 < nb) {
      const double2 d = choose(j + 1, lr == p ? tj[j + 1] : fma(-Aj[lr][j], tj[j + 1], Aj[lr][j + 1]));
      const int pn = __double2loint(d.y);
      const double y = fma(-Aj[pn][j], tj[lr], lr == j ? 0.0 : Aj[pn][lr]);
      if (lane < NP) trow[~j & 1][lane] = lane == j + 1 ? d.x : y * d.x;
    }
    const double t = tj[gc];
    An[gr][gc] = gr == p ? t : fma(-Aj[gr][j], t, gc == j ? 0.0 : Aj[gr][gc]);
    __syncthreads();
  }
  const bool in = gr < nb && gc < nb;
  pinv[fid * NP * NP + (in ? row_piv[gr] * NP + piv_row[gc] : tid)] = in ? A[nb & 1][gr][gc] : 0.0;
#pragma unroll
  for (int u = 0; u < NP * SB / NT; ++u) {
    const int e = tid + u * NT;
    if (e < nb * SB) xr[e] = keep[u];
    if (nb * SB + e < q * SB) xr[nb * SB + e] = moved[u];
  }
}

constexpr int kPanelRows = 8;  // rows per thread: panels of up to 2048 rows (the cross, n = 1024)
// A step's first panel: no row has moved yet.
__device__ __forceinline__ void start_cur(int32_t* cur, int64_t fid, int s, int k,
                                          int k0) {
  if (k == k0)
    for (int p = k0 + threadIdx.x; p < s; p += blockDim.x) cur[fid * s + p] = p;
}
// A kernel of a chain launched to overlap the one before: its blocks wait here. (What the chain
// writes is not read through const __restrict__ pointers: the read-only path may hold lines from
// before the wait.)
__device__ __forceinline__ void chain_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
// One CTA per front: choose nb pivot rows among positions k..s-1 by partial pivoting on the panel
// F[k.., K16]; record the row exchanges, update perm and cur (the position before the step of the
// row now at a position), copy the step's columns of the exchanged rows into xrow, and write the
// inverse of the pivot block. The pivot rows come from a trial elimination of the panel in FP32:
// it only ranks candidate rows by magnitude, while every value the factorisation keeps is computed
// from the FP64 entries. Each thread keeps its panel rows (row tid + t * 256, t < ROWS) in
// registers and each warp publishes its best candidate row to shared memory, so a pivot costs one
// block barrier. Bound by the latency of the 16 pivots, once here (580 cycles each) and once in
// the inversion (1010 cycles each). Measured at the root of 2D n = 512 (1023 rows): 40 -> 21 us a
// panel (before: rows read 128 bytes apart by neighbouring lanes, every thread publishing its row,
// shuffles for the maxima, an FP64 division, three barriers and both halves of [A | I] per pivot of
// the inversion).
template <int ROWS>
__global__ void __launch_bounds__(256) k_nd_panel(const double* fronts, int f, int s,
                                                  int k, int nb, int k0, int sb,
                                                  int32_t* perm,
                                                  int32_t* cur,
                                                  double* xrow,
                                                  double* pinv,
                                                  int32_t* swaps,
                                                  int32_t* err) {
  constexpr int NT = 256, NW = NT / 32;
  __shared__ float st[NT][NP + 1];                     // 256 panel rows on their way to registers
  __shared__ __align__(16) float cand[2][NW][NP + 4];  // each warp's best row, double-buffered
  __shared__ __align__(16) uint2 wb[2][NW];            // its magnitude (bits + 1) and index
  __shared__ int sel[NP];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = s - k;
  const int64_t fid = blockIdx.x;
  const double* F = fronts + fid * f * f;
  chain_start();
  start_cur(cur, fid, s, k, k0);
  float rv[ROWS][NP];
  constexpr int D = ROWS <= 4 ? ROWS : 2;  // groups of 256 rows in flight
  double v[D][NP];
  const int hr = tid / NP, hc = tid % NP;  // half a warp reads one row of the panel
  auto fetch = [&](int t) {
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      const int row = t * NT + hr + u * (NT / NP);
      v[t % D][u] = row < m && hc < nb ? F[(int64_t)(k + row) * f + k + hc] : 0.0;
    }
  };
#pragma unroll
  for (int t = 0; t < D; ++t) fetch(t);
#pragma unroll
  for (int t = 0; t < ROWS; ++t) {
    if (t) __syncthreads();
#pragma unroll
    for (int u = 0; u < NP; ++u) st[hr + u * (NT / NP)][hc] = rank_f32(v[t % D][u]);
    __syncthreads();
    if (t + D < ROWS) fetch(t + D);
#pragma unroll
    for (int c = 0; c < NP; ++c) rv[t][c] = st[tid][c];
  }
  unsigned used = 0;  // bit t: row tid + t NT is a pivot row (or does not exist)
#pragma unroll
  for (int t = 0; t < ROWS; ++t)
    if (tid + t * NT >= m) used |= 1u << t;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    if (j >= nb) break;
    // this thread's candidate for pivot j
    float best = -1.0f;
    int bt = 0;
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      const float a = fabsf(rv[t][j]);
      if (!(used >> t & 1u) && a > best) {
        best = a;
        bt = t;
      }
    }
    // the warp's: the largest magnitude, ties to the lower lane
    const unsigned key = best >= 0.0f ? __float_as_uint(best) + 1u : 0u;
    const unsigned top = __reduce_max_sync(0xffffffffu, key);
    if (lane == __ffs(__ballot_sync(0xffffffffu, key == top)) - 1) {
#pragma unroll
      for (int t = 0; t < ROWS; ++t)
        if (t == bt) {
#pragma unroll
          for (int c = 0; c < NP; ++c)
            if (c >= j) cand[j & 1][warp][c] = rv[t][c];
        }
      wb[j & 1][warp] = make_uint2(top, (unsigned)(tid + bt * NT));
    }
    __syncthreads();
    // the block's, ties to the lower warp
    const uint2 mine = wb[j & 1][lane % NW];
    const unsigned bk = __reduce_max_sync(0xffffffffu, mine.x);
    const int bw = __ffs(__ballot_sync(0xffffffffu, mine.x == bk)) - 1;
    const unsigned pr = __shfl_sync(0xffffffffu, mine.y, bw);
    if (bk < 2u || bk > 0x7f800000u || pr >= (unsigned)m) {  // zero, Inf: uniform over the block
      if (tid == 0) {
        atomicOr(err, 2);
        swaps[fid * kSwapInts] = 0;  // the next kernels of the step then exchange nothing
      }
      return;
    }
    if (tid == 0) sel[j] = (int)pr;
    if ((int)(pr % NT) == tid) used |= 1u << (pr / NT);
    float pv[NP];  // the pivot row from column j on
#pragma unroll
    for (int c = 0; c < NP; ++c) pv[c] = c >= j ? cand[j & 1][bw][c] : 0.0f;
    const float ipv = __fdividef(1.0f, pv[j]);  // ranks only
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      if (used >> t & 1u) continue;
      const float l = rv[t][j] * ipv;
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c > j) rv[t][c] = fmaf(-l, pv[c], rv[t][c]);
    }
  }
  __syncthreads();  // sel complete
  panel_tail(F, f, s, k, nb, k0, sb, fid, sel, perm, cur, xrow, pinv, swaps, err);
}

// The same for panels of more than kPanelRows * 256 rows (the root planes of 3D grids): the same
// FP32 trial elimination with the ranking rows in a global scratch (L2-resident) instead of
// registers; each thread handles rows tid + t * 256, t < 64 (up to 16 384 rows).
__global__ void __launch_bounds__(256) k_nd_panel_big(const double* fronts, int f,
                                                      int s, int k, int nb, int k0, int sb,
                                                      int32_t* perm,
                                                      int32_t* cur,
                                                      double* xrow,
                                                      double* pinv,
                                                      int32_t* swaps,
                                                      int32_t* err,
                                                      float* __restrict__ scratch) {
  constexpr int NT = 256, PS = NP + 1;
  __shared__ float cand[2][NT][PS];
  __shared__ float wbest[2][8];
  __shared__ int wbi[2][8];
  __shared__ int sel[NP];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = s - k;
  const int64_t fid = blockIdx.x;
  const double* F = fronts + fid * f * f;
  chain_start();
  start_cur(cur, fid, s, k, k0);
  float* pan = scratch + fid * (int64_t)s * PS;
  const int nrows = (m - tid + NT - 1) / NT;  // rows of this thread (<= 64)
  float best = -1.0f;
  int bt = 0;
  for (int t = 0; t < nrows; ++t) {
    const int i = tid + t * NT;
    const double* Fi = F + (int64_t)(k + i) * f + k;
    double v[NP];
#pragma unroll
    for (int c = 0; c < NP; ++c) v[c] = c < nb ? Fi[c] : 0.0;
#pragma unroll
    for (int c = 0; c < NP; ++c) pan[(int64_t)i * PS + c] = rank_f32(v[c]);
    const float a = fabsf(rank_f32(v[0]));
    if (a > best) {
      best = a;
      bt = t;
    }
  }
  unsigned long long used = 0;
  for (int j = 0; j < nb; ++j) {
    int bi = best >= 0.0f ? tid + bt * NT : m;
    if (best >= 0.0f) {
      const float* rowc = pan + (int64_t)bi * PS;
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c >= j) cand[j & 1][tid][c] = rowc[c];
    }
    warp_argmax_f(best, bi);
    if (lane == 0) {
      wbest[j & 1][warp] = best;
      wbi[j & 1][warp] = bi;
    }
    __syncthreads();
    float b = wbest[j & 1][0];
    int pr = wbi[j & 1][0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) {
      const float bw = wbest[j & 1][w];
      const int iw = wbi[j & 1][w];
      if (bw > b || (bw == b && iw < pr)) {
        b = bw;
        pr = iw;
      }
    }
    if (!(b > 0.0f) || !isfinite(b) || pr >= m) {  // uniform
      if (tid == 0) {
        atomicOr(err, 2);
        swaps[fid * kSwapInts] = 0;
      }
      return;
    }
    if (tid == 0) sel[j] = pr;
    const int owner = pr % NT;
    if (owner == tid) used |= 1ull << (pr / NT);
    float pv[NP];
#pragma unroll
    for (int c = 0; c < NP; ++c) pv[c] = c >= j ? cand[j & 1][owner][c] : 0.0f;
    const float ipv = 1.0f / pv[j];
    best = -1.0f;
    bt = 0;
    for (int t = 0; t < nrows; ++t) {
      if (used >> t & 1ull) continue;
      float* row = pan + (int64_t)(tid + t * NT) * PS;
      float x[NP];
#pragma unroll
      for (int c = 0; c < NP; ++c) x[c] = row[c];
      const float l = x[j] * ipv;
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c > j) x[c] = fmaf(-l, pv[c], x[c]);
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c > j) row[c] = x[c];
      if (j + 1 < nb) {
        float a = 0.0f;
#pragma unroll
        for (int c = 0; c < NP; ++c)
          if (c == j + 1) a = fabsf(x[c]);
        if (a > best) {
          best = a;
          bt = t;
        }
      }
    }
  }
  __syncthreads();  // sel complete
  panel_tail(F, f, s, k, nb, k0, sb, fid, sel, perm, cur, xrow, pinv, swaps, err);
}

// ---- solve ----
// After the factorisation the blocks that a solve reads are stored once more, transposed and
// contiguous per front: FT[m][i] = F[i][m] (m < s, i < f) for the way up, BT[m][i] = F[i][s + m]
// (m < r, i < s) for the way down. Threads that own consecutive rows i then read consecutive
// doubles for every m: no staging, no shuffles, one FMA per element, at every front size. (From
// the row-major fronts a solve at 2D n = 1024 took 1.2 ms: blocks staged in shared memory for
// small fronts, a warp per row with a shuffle reduction for large ones; now 0.66 ms, and 0.14 ms
// instead of 0.23 ms at n = 256.) What bounds it now: the FP64 pipe (2e8 products at n = 1024,
// 0.32 ms; the bytes would take 0.24 ms) and, at the depths above the leaves, the chain of
// launches and gathers; a depth's kernel loads its first matrix values and its indices before it
// waits for the depth before (programmatic dependent launch).
//
// Also stored per eliminated position: where its right-hand side entry comes from (the grid
// point and the children's ring entries of the pivoted row), so that the gather on the way up is
// two loads deep.
constexpr int kTile = 32;
__global__ void __launch_bounds__(256) k_nd_store(const double* __restrict__ fronts, int f, int s,
                                                  int r, const int32_t* __restrict__ E,
                                                  const int32_t* __restrict__ perm,
                                                  const int32_t* __restrict__ inv, int nchild,
                                                  int rc, double* __restrict__ FT,
                                                  double* __restrict__ BT,
                                                  int32_t* __restrict__ gsrc) {
  __shared__ double t[kTile][kTile + 1];
  const int ti = (f + kTile - 1) / kTile, tm = (s + kTile - 1) / kTile;  // tiles of FT
  const int bi = (s + kTile - 1) / kTile, bm = (r + kTile - 1) / kTile;  // tiles of BT
  // one grid dimension for both: fronts (leaves of 2D n = 1024: 65 536) as well as tiles (3D n = 64:
  // 78 864) can exceed the 65 535 blocks of a second one
  const int per = ti * tm + bi * bm + 1;
  const int64_t p = blockIdx.x / per;
  const double* F = fronts + p * f * f;
  const int q0 = blockIdx.x % per;
  int q = q0;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  if (q < ti * tm || (q -= ti * tm) < bi * bm) {
    const bool fwd = q0 < ti * tm;
    const int nr = fwd ? f : s, nm = fwd ? s : r, c0 = fwd ? 0 : s, tr = fwd ? ti : bi;
    const int i0 = (q % tr) * kTile, m0 = (q / tr) * kTile;
    for (int k = y; k < kTile; k += 8)
      if (i0 + k < nr && m0 + x < nm) t[k][x] = F[(int64_t)(i0 + k) * f + c0 + m0 + x];
    __syncthreads();
    double* out = fwd ? FT + p * s * f : BT + p * r * s;
    for (int k = y; k < kTile; k += 8)
      if (m0 + k < nm && i0 + x < nr) out[(int64_t)(m0 + k) * nr + i0 + x] = t[x][k];
    return;
  }
  // gsrc[(p s + m) 3 ..]: grid point, then the children's entries (or -1) of position perm[m]
  for (int m = threadIdx.x; m < s; m += blockDim.x) {
    const int pm = perm[p * s + m];
    int32_t* g = gsrc + (p * s + m) * 3;
    g[0] = E[p * s + pm];
    for (int c = 0; c < 2; ++c) {
      const int a = c < nchild ? inv[(p * f + pm) * 2 + c] : -1;
      g[1 + c] = a < 0 ? -1 : (int32_t)((nchild == 1 ? p : 2 * p + c) * rc + a);
    }
  }
}

struct MvArgs {
  const double* M;      // FT or BT of the depth
  int nr, nm;           // rows i and columns m of a front's block
  int s, r;
  int ib, mg;           // rows per block, groups of threads that split the columns
  const int32_t* src;   // up: gsrc; down: R
  const int32_t* E;     // down: destination points
  const int32_t* inv;   // up: child ring positions of front positions (null at the leaves)
  int nchild, rc;
  const double* uc;     // up: the children's u
  const double* in;     // up: y; down: x (the ancestors' results)
  double* z;            // up: written; down: read
  double* out;          // up: u; down: x
  int wait;             // launched to overlap the kernel before
};

// Up:   w_m = y + children's u, z_i = sum_m F[i][m] w_m (i < s), u_i = children's u + the same sum.
// Down: x_E[i] = z_i - sum_m F[i][s + m] x_R[m].
// Block: ib consecutive rows of one front x mg column groups; group g takes m = g, g + mg, ...,
// and the groups' sums are added in a fixed tree.
template <bool UP>
__global__ void __launch_bounds__(1024) k_nd_mv(MvArgs a) {
  extern __shared__ double sh[];
  double* w = sh;            // nm
  double* part = sh + a.nm;  // ib * mg
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NP = 8;  // values in flight per thread
  const int tid = threadIdx.x, nt = a.ib * a.mg;
  const int ti = tid % a.ib, tm = tid / a.ib, i = blockIdx.y * a.ib + ti;
  const int64_t p = blockIdx.x;  // (a second grid dimension holds 65 535 blocks: too few fronts)
  const double* M = a.M + p * a.nr * a.nm + (i < a.nr ? i : 0);
  const bool live = __any_sync(0xffffffffu, i < a.nr);  // else the warp only helps to gather
  const int nm = live ? a.nm : 0;
  double v[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    const int m = tm + k * a.mg;
    v[k] = m < nm ? __ldg(M + (int64_t)m * a.nr) : 0.0;
  }
  int ca = -1, cb = -1;  // the row's own child entries (up, ring rows)
  if (UP && a.nchild && tm == 0 && i >= a.s && i < a.nr) {
    ca = __ldg(a.inv + (p * a.nr + i) * 2);
    cb = a.nchild > 1 ? __ldg(a.inv + (p * a.nr + i) * 2 + 1) : -1;
  }
  const int m0 = tid < a.nm ? tid : 0;
  int g0 = 0, g1 = -1, g2 = -1;
  if (UP && a.nm) {
    const int32_t* g = a.src + (p * a.s + m0) * 3;
    g0 = __ldg(g);
    g1 = __ldg(g + 1);
    g2 = __ldg(g + 2);
  }
  if (!UP && a.nm) g0 = __ldg(a.src + p * a.r + m0);
  if (a.wait) asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int m = tid; m < a.nm; m += nt) {
    if (m != tid) {
      if (UP) {
        const int32_t* g = a.src + (p * a.s + m) * 3;
        g0 = __ldg(g);
        g1 = __ldg(g + 1);
        g2 = __ldg(g + 2);
      } else {
        g0 = __ldg(a.src + p * a.r + m);
      }
    }
    double t = a.in[g0];
    if (UP && g1 >= 0) t += a.uc[g1];
    if (UP && g2 >= 0) t += a.uc[g2];
    w[m] = t;
  }
  __syncthreads();
  double c0 = 0.0, c1 = 0.0;
  for (int m = tm; m < nm; m += NP * a.mg) {
    double cur[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) cur[k] = v[k];
    const int mn = m + NP * a.mg;
    if (mn < nm) {
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const int mm = mn + k * a.mg;
        v[k] = mm < nm ? __ldg(M + (int64_t)mm * a.nr) : 0.0;
      }
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int mm = m + k * a.mg;
      if (mm >= nm) break;  // the same for a warp's rows of one group
      (k & 1 ? c1 : c0) = fma(cur[k], w[mm], k & 1 ? c1 : c0);
    }
  }
  double acc = c0 + c1;
  if (a.mg > 1) {
    part[tid] = acc;
    __syncthreads();
    for (int h = a.mg >> 1; h > 0; h >>= 1) {
      if (tm < h) {
        acc += part[tid + h * a.ib];
        part[tid] = acc;
      }
      __syncthreads();
    }
  }
  if (tm != 0 || i >= a.nr) return;
  if (UP) {
    if (i < a.s) {
      a.z[p * a.s + i] = acc;
    } else {
      if (ca >= 0) acc += a.uc[(a.nchild == 1 ? p : 2 * p) * a.rc + ca];
      if (cb >= 0) acc += a.uc[(2 * p + 1) * a.rc + cb];
      a.out[p * a.r + (i - a.s)] = acc;
    }
  } else {
    a.out[a.E[p * a.s + i]] = a.z[p * a.s + i] - acc;
  }
}

// y_j = sum_a rows[j][a] u[(j + o_a) mod n], o_a in [-t, t]^d lexicographic (last fastest), or
// y_j = sub_j - that sum. A block's rows are one contiguous span: read coalesced into shared
// memory (odd row width: no bank conflicts), then one thread per point. HBM-bound: 2D n = 1024,
// 88 MB a product; reading each row by its own thread took 54 us, now 29 us.
template <int D, int T>
__global__ void __launch_bounds__(128) k_apply_rows(const double* __restrict__ rows, int logn,
                                                    const double* __restrict__ u,
                                                    const double* sub, double* y, int64_t N,
                                                    int pts) {
  constexpr int W = 2 * T + 1, MU = D == 1 ? W : (D == 2 ? W * W : W * W * W);
  extern __shared__ double sh[];
  const int64_t j0 = (int64_t)blockIdx.x * pts;
  const int np = (int)(N - j0 < pts ? N - j0 : pts);
  for (int e = threadIdx.x; e < np * MU; e += blockDim.x) sh[e] = __ldcs(rows + j0 * MU + e);
  __syncthreads();
  const int64_t mask = ((int64_t)1 << logn) - 1;
  for (int q = threadIdx.x; q < np; q += blockDim.x) {
    const int64_t j = j0 + q;
    int64_t x[D];
    int64_t rem = j;
#pragma unroll
    for (int a = D - 1; a >= 0; --a) {
      x[a] = rem & mask;
      rem >>= logn;
    }
    double acc = 0.0;
#pragma unroll 9
    for (int a = 0; a < MU; ++a) {
      int o = a, off[D];
#pragma unroll
      for (int b = D - 1; b >= 0; --b) {
        off[b] = o % W - T;
        o /= W;
      }
      int64_t col = 0;
#pragma unroll
      for (int b = 0; b < D; ++b) col = (col << logn) | ((x[b] + off[b]) & mask);
      acc = fma(sh[q * MU + a], __ldg(u + col), acc);
    }
    y[j] = sub ? sub[j] - acc : acc;
  }
}

__global__ void k_nd_iota(int32_t* __restrict__ perm, int count, int s) {
  const int64_t total = (int64_t)count * s;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x)
    perm[e] = (int32_t)(e % s);
}

// "<stem>@<depth>": per-depth timer names (stable storage for the timer table)
const char* level_name(const char* stem, int depth) {
  static char names[7][32][24];
  const int k = stem[3] == 'f' ? 0 : stem[3] == 'b' ? 1 : stem[3] == 's' ? 2 : stem[3] == 'a' ? 3
              : stem[3] == 'p' ? 4 : stem[3] == 'r' ? 5 : 6;
  if (depth < 0 || depth >= 32) return stem;
  snprintf(names[k][depth], sizeof names[k][depth], "%s@%d", stem, depth);
  return names[k][depth];
}

int grid_for(int64_t n, int threads) {
  const int64_t b = (n + threads - 1) / threads;
  return (int)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

}  // namespace

cudaError_t launch_nd_assemble(lsp_ctx* c, int depth, const double* rows) {
  NdState& S = *c->nd;
  const NdLevel& lv = S.plan.lv[depth];
  double* F = (double*)S.fronts.p + lv.front_off;
  const int64_t total = (int64_t)lv.count * lv.f * lv.f;
  int t = timer_begin(c, level_name("nd_asm", depth));
  if (lv.nchild == 0) {
    cudaError_t e = cudaMemsetAsync(F, 0, sizeof(double) * total, c->stream);
    if (e != cudaSuccess) return e;
  } else {
    const NdLevel& cl = S.plan.lv[depth + 1];
    k_nd_extend<<<grid_for(total, 256), 256, 0, c->stream>>>(
        F, (const double*)S.fronts.p + cl.front_off, (const int32_t*)S.inv.p + lv.inv_off,
        lv.count, lv.f, lv.nchild, cl.f, cl.s);
  }
  if (lv.asm_n > 0)
    k_nd_scatter<<<grid_for(lv.asm_n, 256), 256, 0, c->stream>>>(
        F, rows, (const int32_t*)S.asm_dst.p + lv.asm_off, (const int32_t*)S.asm_src.p + lv.asm_off,
        lv.asm_n);
  timer_end(c, t);
  return cudaGetLastError();
}

cudaError_t launch_nd_sweep(lsp_ctx* c, int depth) {
  NdState& S = *c->nd;
  const NdLevel& lv = S.plan.lv[depth];
  double* F = (double*)S.fronts.p + lv.front_off;
  int32_t* perm = (int32_t*)S.perm.p + lv.perm_off;
  int32_t* err = (int32_t*)S.err.p;
  if (lv.s == 0) return cudaSuccess;
  int t = timer_begin(c, level_name("nd_sweep", depth));
  if (lv.f <= kNdSmallFront) {
    const size_t smem = sizeof(double) * ((size_t)lv.f * lv.f + 3 * lv.f);
    auto kern = lv.f <= 32   ? k_nd_sweep_small<1>
                : lv.f <= 64 ? k_nd_sweep_small<2>
                : lv.f <= 96 ? k_nd_sweep_small<3>
                : lv.f <= 128 ? k_nd_sweep_small<4> : k_nd_sweep_small<5>;
    // from 113 rows on a front has the SM's shared memory to itself
    kern<<<lv.count, lv.f > 112 ? 512 : 256, smem, c->stream>>>(F, lv.f, lv.s, perm, err);
    timer_end(c, t);
    return cudaGetLastError();
  }
  // blocked steps; perm starts as the identity
  k_nd_iota<<<grid_for((int64_t)lv.count * lv.s, 256), 256, 0, c->stream>>>(perm, lv.count, lv.s);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_nd_blocked(c, depth);
  timer_end(c, t);
  return e;
}

const char* nd_timer_name(int kind, int depth) {
  return level_name(kind == 4 ? "nd_row" : "nd_upd", depth);
}

cudaError_t launch_nd_panel(lsp_ctx* c, int depth, int k, int nb, int k0, int sb) {
  NdState& S = *c->nd;
  const NdLevel& lv = S.plan.lv[depth];
  const double* F = (const double*)S.fronts.p + lv.front_off;
  int32_t* perm = (int32_t*)S.perm.p + lv.perm_off;
  const bool big = lv.s > kPanelRows * 256;
  if (big && !S.pscratch.p) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(lv.count);
  cfg.blockDim = dim3(256);
  cfg.stream = c->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = c->timing ? 0 : 1;
  const int t = timer_begin(c, level_name("nd_pnl", depth));
  cudaError_t e;
  if (big)
    e = cudaLaunchKernelEx(&cfg, k_nd_panel_big, F, lv.f, lv.s, k, nb, k0, sb, perm,
                           (int32_t*)S.cur.p, (double*)S.xrow.p, (double*)S.pinv.p,
                           (int32_t*)S.swaps.p, (int32_t*)S.err.p, (float*)S.pscratch.p);
  else {  // rows per thread: as few as cover the rows that are left
    const int per = (lv.s - k + 255) / 256;
    auto kern = per <= 1 ? k_nd_panel<1> : per <= 2 ? k_nd_panel<2>
                : per <= 4 ? k_nd_panel<4> : k_nd_panel<kPanelRows>;
    e = cudaLaunchKernelEx(&cfg, kern, F, lv.f, lv.s, k, nb, k0, sb, perm, (int32_t*)S.cur.p,
                           (double*)S.xrow.p, (double*)S.pinv.p, (int32_t*)S.swaps.p,
                           (int32_t*)S.err.p);
  }
  timer_end(c, t);
  return e;
}

// The solve's copies of one depth's blocks, after its sweep.
cudaError_t launch_nd_store(lsp_ctx* c, int depth) {
  NdState& S = *c->nd;
  const NdLevel& lv = S.plan.lv[depth];
  if (lv.s == 0) return cudaSuccess;
  const int tf = (lv.f + kTile - 1) / kTile, ts = (lv.s + kTile - 1) / kTile;
  const int tr = (lv.r + kTile - 1) / kTile;
  int t = timer_begin(c, level_name("nd_asm", depth));
  k_nd_store<<<(unsigned)((int64_t)lv.count * (tf * ts + ts * tr + 1)), 256, 0, c->stream>>>(
      (const double*)S.fronts.p + lv.front_off, lv.f, lv.s, lv.r,
      (const int32_t*)S.E.p + lv.E_off, (const int32_t*)S.perm.p + lv.perm_off,
      lv.nchild ? (const int32_t*)S.inv.p + lv.inv_off : nullptr, lv.nchild,
      lv.nchild ? S.plan.lv[depth + 1].r : 0, (double*)S.solve.p + lv.ft_off,
      (double*)S.solve.p + lv.bt_off, (int32_t*)S.gsrc.p + 3 * lv.z_off);
  timer_end(c, t);
  return cudaGetLastError();
}

cudaError_t launch_nd_solve(lsp_ctx* c, const double* y, double* x) {
  NdState& S = *c->nd;
  const NdPlan& P = S.plan;
  const int L = (int)P.lv.size();
  const double* sv = (const double*)S.solve.p;
  double* z = (double*)S.z.p;
  double* u = (double*)S.u.p;
  auto launch = [&](bool up, MvArgs& a, int count) -> cudaError_t {
    // Rows per block: all of a short front (whole warps), else 128 down to 16 until there are two
    // blocks per SM. Column groups: at least eight columns each, until the depth has 512 threads
    // per SM: the next depth's blocks then find room to load beside it (a solve at 2D n = 1024,
    // 256 and 3D n = 32: 660, 140, 222 us; with 2048 threads per SM 752, 149, 251 us).
    auto blocks = [&]() { return (int64_t)count * ((a.nr + a.ib - 1) / a.ib); };
    a.ib = a.nr >= 128 ? 128 : (a.nr + 31) / 32 * 32;
    if (blocks() < 2 * 152) {
      a.ib = 128;
      while (a.ib > 16 && (a.ib >= 2 * a.nr || blocks() < 2 * 152)) a.ib >>= 1;
    }
    a.mg = 1;
    while (2 * a.mg * a.ib <= 1024 && a.nm >= 16 * a.mg &&
           blocks() * a.ib * a.mg < (int64_t)152 * 512)
      a.mg <<= 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(count, (a.nr + a.ib - 1) / a.ib);
    cfg.blockDim = dim3(a.ib * a.mg);
    cfg.dynamicSmemBytes = sizeof(double) * ((size_t)a.nm + (a.mg > 1 ? a.ib * a.mg : 0));
    cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = a.wait ? 1 : 0;
    return up ? cudaLaunchKernelEx(&cfg, k_nd_mv<true>, a)
              : cudaLaunchKernelEx(&cfg, k_nd_mv<false>, a);
  };
  MvArgs a;
  a.wait = 0;  // the first kernel starts after whatever produced y
  for (int d = L - 1; d >= 0; --d) {
    const NdLevel& lv = P.lv[d];
    const NdLevel* cl = lv.nchild ? &P.lv[d + 1] : nullptr;
    if (lv.f == 0) continue;
    int t = timer_begin(c, level_name("nd_fwd", d));
    a.M = sv + lv.ft_off;
    a.nr = lv.f;
    a.nm = lv.s;
    a.s = lv.s;
    a.r = lv.r;
    a.src = (const int32_t*)S.gsrc.p + 3 * lv.z_off;
    a.E = nullptr;
    a.inv = lv.nchild ? (const int32_t*)S.inv.p + lv.inv_off : nullptr;
    a.nchild = lv.nchild;
    a.rc = cl ? cl->r : 0;
    a.uc = cl ? u + cl->u_off : nullptr;
    a.in = y;
    a.z = z + lv.z_off;
    a.out = u + lv.u_off;
    const cudaError_t e = launch(true, a, lv.count);
    if (e != cudaSuccess) return e;
    timer_end(c, t);
    a.wait = !c->timing;
  }
  for (int d = 0; d < L; ++d) {
    const NdLevel& lv = P.lv[d];
    if (lv.s == 0) continue;
    int t = timer_begin(c, level_name("nd_bwd", d));
    a.M = sv + lv.bt_off;
    a.nr = lv.s;
    a.nm = lv.r;
    a.s = lv.s;
    a.r = lv.r;
    a.src = (const int32_t*)S.R.p + lv.R_off;
    a.E = (const int32_t*)S.E.p + lv.E_off;
    a.inv = nullptr;
    a.nchild = 0;
    a.rc = 0;
    a.uc = nullptr;
    a.in = x;
    a.z = z + lv.z_off;
    a.out = x;
    const cudaError_t e = launch(false, a, lv.count);
    if (e != cudaSuccess) return e;
    timer_end(c, t);
  }
  return cudaGetLastError();
}

// Dynamic shared memory up to what a block can have, for the kernels whose need varies with the
// plan. The limit belongs to the kernel, not to a context: one set to a plan's need would be lowered
// by the next, smaller plan of another context, whose launches are then refused.
cudaError_t nd_prepare_kernels() {
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  auto allow = [&](auto kern) {
    cudaFuncAttributes at;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, kern);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               most - (int)at.sharedSizeBytes);
  };
  allow(k_nd_mv<true>);
  allow(k_nd_mv<false>);
  allow(k_nd_sweep_small<1>);
  allow(k_nd_sweep_small<2>);
  allow(k_nd_sweep_small<3>);
  allow(k_nd_sweep_small<4>);
  allow(k_nd_sweep_small<5>);
  return e;
}

cudaError_t launch_apply_rows(lsp_ctx* c, const double* rows, int mu, int t, const double* u,
                              double* y, const double* sub) {
  const int64_t N = c->geo.N;
  const int d = c->geo.d;
  int logn = 0;
  while ((1 << logn) < c->geo.n) ++logn;
  const int pts = mu > 27 ? 32 : 128;
  const size_t smem = sizeof(double) * mu * pts;  // at most 32 KiB
  int tm = timer_begin(c, "apply_rows");
  auto go = [&](auto kern) {
    kern<<<(unsigned)((N + pts - 1) / pts), 128, smem, c->stream>>>(rows, logn, u, sub, y, N, pts);
  };
  if (d == 1)
    go(k_apply_rows<1, 1>);
  else if (d == 2)
    t == 1 ? go(k_apply_rows<2, 1>) : go(k_apply_rows<2, 2>);
  else
    t == 1 ? go(k_apply_rows<3, 1>) : go(k_apply_rows<3, 2>);
  timer_end(c, tm);
  return cudaGetLastError();
}

}  // namespace lsp
