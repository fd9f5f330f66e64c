// Partial inversion of the large fronts (f > kNdSmallFront) of the nested dissection, in steps of
// kNdStep = 64 pivots (see nd.h for the front layout and k_nd.cu for the panels). A step makes the
// columns K = [k0, k0 + sb) of a front the final ones in sub-steps q of 16 pivots K_q, each of which
// touches only the columns of K from K_q on: the panel chooses the pivot rows and inverts the
// 16 x 16 pivot block, k_nd_sub forms V_q (-F[., K_q] A_q^-1; A_q^-1 on the pivot rows), which
// takes the place of F[., K_q], and applies it to the columns of K to the right. Everything else
// is then updated at once,
//   F[i, j] <- (i in K_q, q > p(j) ? 0 : F[i, j]) + sum_{q > p(j)} V_q[i, :] W_q[:, j]
// with p(j) = -1 outside K, p for j in K_p; W_q: the pivot rows of K_q as the sub-steps before it
// leave them (k_nd_wsplit); V_q = 0 on the pivot rows of later sub-steps (their part of the sum is
// in W already). These are the products of the elimination by 16 pivots at a time; one product
// with the inverse of the whole 64 x 64 block would be cheaper, but was measured to lose a digit of
// the solution (2D n = 1024).
//
// The sum is FP64 work that the FP64 pipe would bound (1.25 TFLOP/s): it runs on the tensor cores
// instead, by an error-free split (the scheme of Ozaki, Ogita, Oishi and Rump for matrix products
// from exact partial products): every row of V and every column of W is scaled by a power of two and
// written as seven digits to base 512, balanced in [-256, 255], which f16 holds exactly; products
// of digits and their sums over 64 terms and up to four pairs of equal weight are integers up to
// 2^24, exact in the FP32 accumulators (with five to seven pairs a sum beyond 2^24 may be rounded,
// by less than 2^-57 of the result). The 28 digit products whose weight reaches 2^-54 of the leading
// one are formed, put together as one integer, rounded once to FP64 and added: entries down to 2^-9
// of the largest of their row and column are not rounded at all by the split. With digits for
// 55 bits the solution lost a digit in 3D, where rows and columns decay.
//
// What bounds it: per 128 x 64 tile 224 products of 128 x 32 x 16 (47 cycles each with both operands
// in shared memory) beside about 80 integer operations and one FP64 addition per entry to take the
// sums out: 14e3 cycles, against 262e3 of the FP64 pipe.
// Measured against rank-16 updates of the whole front on the FP64 pipe: the updates of 3D n = 32
// about 100 -> 6 ms, the whole factorisation 118 -> 23 ms, of 2D n = 512 28.4 -> 13.4 ms; the
// unrefined backward error is smaller (3D) or equal (2D).
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>

#include "digits.cuh"
#include "nd.h"
#include "tc_common.cuh"

namespace lsp {
namespace {

constexpr int NP = kNdPanel, SB = kNdStep;
constexpr int kTileJ = 128, kTileI = 64;  // columns (tensor-memory lanes) x rows of a tile
constexpr int kBytesW = kTileJ * SB * 2, kBytesU = kTileI * SB * 2;  // one digit of a tile

// One kernel of a chain launched to overlap. What an earlier kernel of the chain writes is read
// through plain pointers: a const __restrict__ one allows loads through the read-only path, whose
// lines may date from before the wait.
__device__ __forceinline__ void chain_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Position, before the step, of the row that is at position x now (only positions in [k0, s) move).
__device__ __forceinline__ int row_id(const int32_t* cu, int x, int k0, int s) {
  return x >= k0 && x < s ? cu[x] : x;
}

// Sub-step: kSubRows rows of one front per block. With the row exchanges of the panel (position dst
// takes the row that was at src; the panel left the exchanged rows' 64 columns in xrow, the pivot
// rows first), V = -C A^-1 (A^-1 on the pivot rows), F[x, K16] = V, F[x, j] += V W16[:, j] for
// the columns of the step to the right. Blocks read only xrow and their own rows. V is kept for the
// update, under the row's position before the step. Bound by the FP64 pipe (640 multiply-adds a row on
// average); eight rows a block spread the fronts of about a thousand rows over all SMs.
constexpr int kSubRows = 8;
__global__ void __launch_bounds__(128) k_nd_sub(double* __restrict__ fronts, int f, int s, int k,
                                                int nb, int k0, int sb,
                                                const double* xrow,
                                                const double* pinv,
                                                const int32_t* swaps,
                                                const int32_t* cur,
                                                double* __restrict__ vst) {
  __shared__ double C[kSubRows][SB + 1], W[NP][SB], V[kSubRows][NP + 1], pi[NP][NP];
  __shared__ int from[kSubRows];  // index in xrow, or -1: the row is where it was
  chain_start();
  const int tid = threadIdx.x, x0 = blockIdx.x * kSubRows;
  const int64_t fid = blockIdx.y;
  double* F = fronts + fid * f * f;
  const int32_t* sw = swaps + fid * kNdSwapInts;
  const double* xr = xrow + fid * (2 * NP * SB);
  const int vr = tid / NP, vc = tid % NP;  // 128 threads = 8 rows x 16 columns of V
  const int id = x0 + vr < f ? row_id(cur + fid * s, x0 + vr, k0, s) : 0;
  if (tid < kSubRows) from[tid] = -1;
  __syncthreads();
  if (tid < 2 * NP) {
    const int at = sw[1 + tid] - x0;
    if (tid < sw[0] && at >= 0 && at < kSubRows) from[at] = tid;
  }
#pragma unroll
  for (int e = tid; e < NP * NP; e += 128) pi[e / NP][e % NP] = pinv[fid * NP * NP + e];
#pragma unroll
  for (int e = tid; e < NP * SB; e += 128) W[e / SB][e % SB] = e / SB < nb ? xr[e] : 0.0;
  __syncthreads();
#pragma unroll
  for (int e = tid; e < kSubRows * SB; e += 128) {
    const int r = e / SB, c = e % SB, x = x0 + r;
    C[r][c] = x < f && c < sb ? (from[r] >= 0 ? xr[from[r] * SB + c] : F[(int64_t)x * f + k0 + c])
                              : 0.0;
  }
  __syncthreads();
  const int kc = k - k0;  // first column of the sub-step within the step
  {
    const int x = x0 + vr;
    double a = 0.0;
    if (x >= k && x < k + nb) {
      a = pi[x - k][vc];
    } else {
#pragma unroll
      for (int m = 0; m < NP; ++m) a = fma(m < nb ? C[vr][kc + m] : 0.0, pi[m][vc], a);
      a = -a;
    }
    V[vr][vc] = a;
    if (x < f) vst[(fid * f + id) * SB + kc + vc] = a;
  }
  __syncthreads();
#pragma unroll
  for (int e = tid; e < kSubRows * SB; e += 128) {
    const int r = e / SB, c = e % SB, x = x0 + r;
    if (x >= f || c >= sb) continue;
    double a = C[r][c];
    if (c >= kc + nb) {
      if (x >= k && x < k + nb) a = 0.0;
#pragma unroll
      for (int m = 0; m < NP; ++m) a = fma(V[r][m], W[m][c], a);
    } else if (c >= kc) {
      a = V[r][c - kc];
    }
    F[(int64_t)x * f + k0 + c] = a;
  }
}

__device__ __forceinline__ uint32_t pack_f16(int a, int b) {
  const __half2 h = __floats2half2_rn((float)a, (float)b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// Eight consecutive values (K indices) of one row of a digit tile, all digits.
__device__ __forceinline__ void store_digits(const double (&v)[8], int e, uint8_t* tile, int bytes,
                                             int row, int kk) {
  uint32_t w[kDigits][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    int a[kDigits], b[kDigits];
    digits_of(v[2 * p], e, a);
    digits_of(v[2 * p + 1], e, b);
#pragma unroll
    for (int t = 0; t < kDigits; ++t) w[t][p] = pack_f16(a[t], b[t]);
  }
#pragma unroll
  for (int t = 0; t < kDigits; ++t)
    *reinterpret_cast<uint4*>(tile + t * bytes + tc::kmajor_off(row, kk, SB)) =
        make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
}

// W: eight columns of one front per block, one thread per column and pivot row of a sub-step. The
// pivot rows' entries (at cur[k0 + a], their positions before the step) go through the elimination
// by the sub-steps before their own, W_q += sum_{p < q} V_p[K_q] W_p (bound by the FP64 pipe, 1536
// multiply-adds a column), and become digits; then the rows that the step's exchanges moved to
// positions outside K are moved in these columns (they come from positions in K, which the update
// overwrites).
constexpr int kSplitCols = 8;
__global__ void __launch_bounds__(128) k_nd_wsplit(double* __restrict__ fronts, int f, int s, int k0,
                                                   int sb, int nj, const int32_t* cur,
                                                   const double* vst,
                                                   uint8_t* __restrict__ digits,
                                                   int32_t* __restrict__ expo) {
  __shared__ double W[SB][kSplitCols + 1], L[SB - NP][SB - NP + 1];  // L[a - 16][c] = V_p[row a]
  __shared__ int src[SB], mdst[SB], msrc[SB], nmove;
  chain_start();
  const int tid = threadIdx.x;
  const int64_t fid = blockIdx.y;
  double* F = fronts + fid * f * f;
  const int32_t* cu = cur + fid * s;
  if (tid == 0) nmove = 0;
  if (tid < SB) src[tid] = tid < sb ? cu[k0 + tid] : 0;
  __syncthreads();
  const int j0 = blockIdx.x * kSplitCols;
#pragma unroll
  for (int u = 0; u < SB * kSplitCols / 128; ++u) {
    const int a = (tid + u * 128) / kSplitCols, j = j0 + tid % kSplitCols;
    const int jk = j - k0;  // a column of K_p starts as V_p, below its own sub-step
    double w = 0.0;
    if (a < sb && j < f) {
      if (jk < 0 || jk >= sb)
        w = F[(int64_t)src[a] * f + j];
      else if (a / NP > jk / NP)
        w = vst[(fid * f + src[a]) * SB + jk];
    }
    W[a][tid % kSplitCols] = w;
  }
#pragma unroll 6
  for (int e = tid; e < (SB - NP) * (SB - NP); e += 128) {
    const int a = e / (SB - NP), c = e % (SB - NP);
    L[a][c] = a + NP < sb && c < (a + NP) / NP * NP ? vst[(fid * f + src[a + NP]) * SB + c] : 0.0;
  }
  for (int p = k0 + sb + tid; p < s; p += 128) {
    const int c = cu[p];
    if (c != p) {
      const int a = atomicAdd(&nmove, 1);
      if (a < SB) {
        mdst[a] = p;
        msrc[a] = c;
      }
    }
  }
  __syncthreads();
  {
    const int r = tid / kSplitCols, j = tid % kSplitCols;
#pragma unroll
    for (int q = 1; q < SB / NP; ++q) {
      double a = W[q * NP + r][j];
#pragma unroll
      for (int c = 0; c < q * NP; ++c) a = fma(L[(q - 1) * NP + r][c], W[c][j], a);
      W[q * NP + r][j] = a;
      __syncthreads();
    }
  }
  if (tid < SB) {  // eight lanes per column: eight pivots each
    const int jj = tid / 8, g = tid % 8, j = j0 + jj;
    double v[8];
    int e = kExpNone;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = W[g * 8 + u][jj];
      e = max(e, exp_of(v[u]));
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    uint8_t* tile = digits + (fid * nj + j / kTileJ) * (int64_t)(kDigits * kBytesW);
    store_digits(v, e, tile, kBytesW, j % kTileJ, g * 8);
    if (g == 0 && j < f) expo[fid * f + j] = e;
  }
  const int n = min(nmove, SB);
  for (int e = tid; e < n * kSplitCols; e += 128) {
    const int a = e / kSplitCols, j = j0 + e % kSplitCols;
    if (j < f && (j < k0 || j >= k0 + sb))
      F[(int64_t)mdst[a] * f + j] = F[(int64_t)msrc[a] * f + j];
  }
}

// V: 64 rows per block, four threads per row (one per sub-step).
__global__ void __launch_bounds__(256) k_nd_vsplit(int f, int s, int k0, int sb,
                                                   const int32_t* cur,
                                                   const double* vst,
                                                   uint8_t* __restrict__ digits,
                                                   int32_t* __restrict__ expo) {
  chain_start();
  const int tid = threadIdx.x, row = tid >> 2, part = tid & 3;
  const int64_t fid = blockIdx.y;
  const int i = blockIdx.x * kTileI + row;
  const int id = i < f ? row_id(cur + fid * s, i, k0, s) : 0;
  const double* Vi = vst + (fid * f + id) * SB;
  // a pivot row of K takes part from its own sub-step on
  const bool on = i < f && (i < k0 || i >= k0 + sb || part >= (i - k0) / NP);
  double v[2][8];
  int e = kExpNone;
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int c = part * 16 + g * 8 + q;
      v[g][q] = on && c < sb ? Vi[c] : 0.0;
      e = max(e, exp_of(v[g][q]));
    }
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
  uint8_t* tile = digits + (fid * gridDim.x + blockIdx.x) * (int64_t)(kDigits * kBytesU);
#pragma unroll
  for (int g = 0; g < 2; ++g) store_digits(v[g], e, tile, kBytesU, row, part * 16 + g * 8);
  if (part == 0 && i < f) expo[fid * f + i] = e;
}

// 4 consecutive FP32 columns of this thread's tensor-memory lane, without waiting.
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// The update. One block per SM takes a run of the 128 x 64 tiles (columns j x rows i) of all fronts,
// rows fastest: the seven W digit tiles stay in shared memory while the columns stay the same, the
// V digit tiles have two buffers. The last warp copies the tiles and issues the 28 digit products
// of one half of the rows at a time, weight l = t + t' into accumulator columns 256 half + 32 l
// (unrolled, descriptors by one addition: a loop took 109 cycles a product to issue; from one lane
// of a branch, without uniform registers, 57 to 79). The other sixteen warps take the sums of one
// half out (8 rows each, the entries to update loaded a half ahead) while the products of the other
// run. Cycles a half: products 5.3e3 (47 each: shared-memory reads of the operands), sums 4e3 and
// 2e3 of loads; the two sides meet at about 7e3. The products one after the other with the sums,
// 64 rows at a time: 25e3 a tile.
constexpr int kSumWarps = 16, kGemmThreads = 32 * (kSumWarps + 1);
constexpr int kHalf = kTileI / 2, kWarpRows = kHalf / (kSumWarps / 4);
constexpr size_t kGemmSmem = (size_t)kDigits * (kBytesW + 2 * kBytesU);
__global__ void __launch_bounds__(kGemmThreads, 1) k_nd_gemm(
    double* __restrict__ fronts, int f, int k0, int sb, int64_t total, const uint8_t* dW,
    const int32_t* eW, const uint8_t* dV, const int32_t* eV, int32_t* __restrict__ err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t bar_w, bar_v[2], bar_mma[2], bar_free[2];
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int ni = (f + kTileI - 1) / kTileI, nj = (f + kTileJ - 1) / kTileJ;
  const int64_t g0 = total * blockIdx.x / gridDim.x, g1 = total * (blockIdx.x + 1) / gridDim.x;
  const int nt = (int)(g1 - g0);
  if (tid == 0) {
    tc::mbar_init(&bar_w, 1);
    for (int h = 0; h < 2; ++h) {
      tc::mbar_init(&bar_v[h], 1);
      tc::mbar_init(&bar_mma[h], 1);
      tc::mbar_init(&bar_free[h], kSumWarps);
    }
  }
  if (warp == 0) tc::tmem_alloc(&tslot, 512);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tslot;
  chain_start();
  // a tile's place: row tile, column tile, front
  int ti = (int)(g0 % ni), tj = (int)(g0 / ni % nj);
  int64_t fid = g0 / ni / nj;
  auto advance = [&]() {
    if (++ti == ni) {
      ti = 0;
      if (++tj == nj) {
        tj = 0;
        ++fid;
      }
    }
  };
  if (warp == kSumWarps) {
    if (nt > 0) {
      uint8_t* sW = smem;
      uint8_t* sV = smem + kDigits * kBytesW;
      int loads_w = 0, loads_v = 0, sets = 0;
      auto load_w = [&]() {
        if (lane == 0) {
          tc::mbar_expect_tx(&bar_w, kDigits * kBytesW);
          tc::bulk_g2s(sW, dW + (fid * nj + tj) * (kDigits * kBytesW), kDigits * kBytesW, &bar_w);
        }
        __syncwarp();
        ++loads_w;
      };
      auto load_v = [&]() {
        const int b = loads_v++ & 1;
        if (lane == 0) {
          tc::mbar_expect_tx(&bar_v[b], kDigits * kBytesU);
          tc::bulk_g2s(sV + b * (kDigits * kBytesU), dV + (fid * ni + ti) * (kDigits * kBytesU),
                       kDigits * kBytesU, &bar_v[b]);
        }
        __syncwarp();
      };
      auto wait = [&](uint64_t* bar, uint32_t phase) {  // every lane asks
        return __all_sync(0xffffffffu, tc::mbar_wait(bar, phase, err, kNdErrWait)) != 0;
      };
      const int ksteps = (sb + 15) / 16;
      constexpr uint32_t sbo = (SB / 8) * 128;
      constexpr uint32_t idesc = tc::idesc_f16(kTileJ, kHalf);
      const uint64_t da = tc::desc_kmajor(tc::smem_u32(sW), 128, sbo);
      load_w();
      load_v();
      bool ok = true;
      for (int t = 0; ok && t < nt; ++t) {
        const uint64_t dv =
            tc::desc_kmajor(tc::smem_u32(sV + (t & 1) * (kDigits * kBytesU)), 128, sbo);
        const uint32_t before = (uint32_t)(t - 1) & 1u;  // the tile before's phase of bar_free
        for (int h = 0; ok && h < 2; ++h) {
          // once the sums of the half before in these accumulators are out, its products are done
          if (t > 0) ok = wait(&bar_free[h], before);
          if (h == 0) {
            if (ok && t > 0 && ti == 0) {  // other columns: all products on W must be done
              ok = wait(&bar_free[1], before);
              if (ok) load_w();
            }
            // (a phase of W passed already returns at once)
            ok = ok && wait(&bar_w, (uint32_t)(loads_w - 1) & 1u) &&
                 wait(&bar_v[t & 1], (uint32_t)(t >> 1) & 1u);
          }
          if (!ok) break;
          if (h == 1) {  // the tile before is done with the other V buffer
            advance();
            if (t + 1 < nt) load_v();
          }
          tc::fence_after();
          const uint64_t db = dv + (uint64_t)(h * (kHalf / 8) * sbo / 16);
          const uint32_t acc = tmem + (uint32_t)(h * 256);
          if (ksteps == SB / 16) {
#pragma unroll
            for (int a = 0; a < kDigits; ++a)
#pragma unroll
              for (int b = 0; a + b < kLevels; ++b)
#pragma unroll
                for (int q = 0; q < SB / 16; ++q)
                  tc::mma_bf16_warp(acc + (uint32_t)((a + b) * kHalf),
                                    da + (uint64_t)(a * kBytesW / 16 + 16 * q),
                                    db + (uint64_t)(b * kBytesU / 16 + 16 * q), idesc,
                                    (a > 0 || q > 0) ? 1u : 0u);
          } else {
            for (int a = 0; a < kDigits; ++a)
              for (int b = 0; a + b < kLevels; ++b)
                for (int q = 0; q < ksteps; ++q)
                  tc::mma_bf16_warp(acc + (uint32_t)((a + b) * kHalf),
                                    da + (uint64_t)(a * kBytesW / 16 + 16 * q),
                                    db + (uint64_t)(b * kBytesU / 16 + 16 * q), idesc,
                                    (a > 0 || q > 0) ? 1u : 0u);
          }
          tc::commit_warp(&bar_mma[h]);
          ++sets;
        }
      }
      // before leaving (after a wait that gave up as well): copies and products in flight
      tc::mbar_wait(&bar_w, (uint32_t)(loads_w - 1) & 1u, err, 0);
      for (int b = 0; b < 2; ++b) {
        const int uses = loads_v / 2 + (b < loads_v % 2 ? 1 : 0);
        if (uses) tc::mbar_wait(&bar_v[b], (uint32_t)(uses - 1) & 1u, err, 0);
        const int n = sets / 2 + (b < sets % 2 ? 1 : 0);
        if (n) tc::mbar_wait(&bar_mma[b], (uint32_t)(n - 1) & 1u, err, 0);
      }
    }
  } else if (nt > 0) {
    const int zhi = k0 + sb, cj = (warp & 3) * 32 + lane, ci = (warp >> 2) * kWarpRows;
    // Entries to update of half h of the tile (ti, tj, fid), and its exponents. Rows below zlo and
    // from zhi on keep their entry: the pivot rows of sub-steps after the column's own (all of K
    // for a column outside K) are replaced.
    double old[kWarpRows], nxt[kWarpRows];
    int ej = 0, er = 0;  // exponent of the column; of row lane % 8
    auto fetch = [&](int h, double (&o)[kWarpRows], int& ec, int& ex) {
      const int j = tj * kTileJ + cj, ib = ti * kTileI + h * kHalf + ci;
      const bool jl = j < f;
      const int zlo = jl && j >= k0 && j < zhi ? k0 + ((j - k0) / NP + 1) * NP : k0;
      const double* Fj = fronts + (fid * f + ib) * f + j;
#pragma unroll
      for (int q = 0; q < kWarpRows; ++q) {
        const int i = ib + q;
        o[q] = jl && i < f && (i < zlo || i >= zhi) ? Fj[(int64_t)q * f] : 0.0;
      }
      ec = jl ? eW[fid * f + j] : kExpNone;
      ex = ib + (lane & 7) < f ? eV[fid * f + ib + (lane & 7)] : kExpNone;
    };
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)ci;
    bool ok = true;
    fetch(0, old, ej, er);
    for (int u = 0; u < 2 * nt; ++u) {
      const int h = u & 1, j = tj * kTileJ + cj, ib = ti * kTileI + h * kHalf + ci;
      double* Fj = fronts + (fid * f + ib) * f + j;
      const int rows = j < f ? f - ib : 0;  // that exist
      // (one lane asks, the others follow its answer)
      const bool got =
          lane == 0 ? tc::mbar_wait(&bar_mma[h], (uint32_t)(u >> 1) & 1u, err, kNdErrWait) : true;
      ok = __all_sync(0xffffffffu, got);
      if (!ok) break;
      tc::fence_after();
      int ejn = 0, ern = 0;
#pragma unroll
      for (int c0 = 0; c0 < kWarpRows; c0 += 4) {
        uint32_t r[kLevels][4];
#pragma unroll
        for (int l = 0; l < kLevels; ++l)
          tmem_ld4(taddr + (uint32_t)(h * 256 + l * kHalf + c0), r[l]);
        if (c0 == 0) {
          if (h == 1) advance();
          if (u + 1 < 2 * nt) fetch(h ^ 1, nxt, ejn, ern);
        }
        tc::ld_wait();
        if (c0 + 4 == kWarpRows) {
          tc::fence_before();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&bar_free[h]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          int a[kLevels];
#pragma unroll
          for (int l = 0; l < kLevels; ++l) a[l] = __float2int_rn(__uint_as_float(r[l][q]));
          const double v = sum_of(a, __shfl_sync(0xffffffffu, er, c0 + q) + ej - 16);
          if (c0 + q < rows) Fj[(int64_t)(c0 + q) * f] = old[c0 + q] + v;
        }
      }
#pragma unroll
      for (int q = 0; q < kWarpRows; ++q) old[q] = nxt[q];
      ej = ejn;
      er = ern;
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace

int64_t nd_tc_bytes_w(int f) { return (int64_t)((f + kTileJ - 1) / kTileJ) * kDigits * kBytesW; }
int64_t nd_tc_bytes_u(int f) { return (int64_t)((f + kTileI - 1) / kTileI) * kDigits * kBytesU; }

cudaError_t nd_tc_prepare() {
  return cudaFuncSetAttribute(k_nd_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kGemmSmem);
}

// Blocked partial inversion of the fronts of one depth (perm holds the identity).
cudaError_t launch_nd_blocked(lsp_ctx* c, int depth) {
  NdState& S = *c->nd;
  const NdLevel& lv = S.plan.lv[depth];
  double* F = (double*)S.fronts.p + lv.front_off;
  const int f = lv.f, s = lv.s, count = lv.count;
  int32_t* err = (int32_t*)S.err.p;
  int32_t* cur = (int32_t*)S.cur.p;
  double* xrow = (double*)S.xrow.p;
  double* pinv = (double*)S.pinv.p;
  int32_t* swaps = (int32_t*)S.swaps.p;
  uint8_t* dW = (uint8_t*)S.digits.p;
  uint8_t* dV = dW + (int64_t)count * nd_tc_bytes_w(f);
  double* vst = (double*)S.vst.p;
  int32_t* eW = (int32_t*)S.expo.p;
  int32_t* eV = eW + (int64_t)count * f;
  const int nj = (f + kTileJ - 1) / kTileJ, ni = (f + kTileI - 1) / kTileI;
  const int64_t total = (int64_t)count * nj * ni;
  const int blocks = (int)std::min<int64_t>(total, 152);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  auto go = [&](auto kern, dim3 grid, int threads, size_t smem, auto... args) -> cudaError_t {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cfg.attrs = at;
    cfg.numAttrs = c->timing ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
  };
  cudaError_t e;
  for (int k0 = 0; k0 < s; k0 += SB) {
    const int sb = std::min(SB, s - k0);
    for (int k = k0; k < k0 + sb; k += NP) {
      const int nb = std::min(NP, k0 + sb - k);
      if ((e = launch_nd_panel(c, depth, k, nb, k0, sb)) != cudaSuccess) return e;
      const int t = timer_begin(c, nd_timer_name(4, depth));
      e = go(k_nd_sub, dim3((f + kSubRows - 1) / kSubRows, count), 128, 0, F, f, s, k, nb, k0,
             sb, (const double*)xrow, (const double*)pinv, (const int32_t*)swaps,
             (const int32_t*)cur, vst);
      if (e != cudaSuccess) return e;
      timer_end(c, t);
    }
    int t = timer_begin(c, nd_timer_name(4, depth));
    e = go(k_nd_wsplit, dim3((f + kSplitCols - 1) / kSplitCols, count), 128, 0, F, f, s, k0, sb, nj,
           (const int32_t*)cur, (const double*)vst, dW, eW);
    if (e == cudaSuccess)
      e = go(k_nd_vsplit, dim3(ni, count), 256, 0, f, s, k0, sb, (const int32_t*)cur,
             (const double*)vst, dV, eV);
    if (e != cudaSuccess) return e;
    timer_end(c, t);
    t = timer_begin(c, nd_timer_name(5, depth));
    e = go(k_nd_gemm, dim3(blocks), kGemmThreads, kGemmSmem, F, f, k0, sb, total,
           (const uint8_t*)dW, (const int32_t*)eW, (const uint8_t*)dV, (const int32_t*)eV, err);
    if (e != cudaSuccess) return e;
    timer_end(c, t);
  }
  return cudaSuccess;
}

}  // namespace lsp
