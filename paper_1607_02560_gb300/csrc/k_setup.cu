// Steps a1-a2 and the domain bookkeeping of a3:
//  * potential statistics v_min, v_max, mean (Sec. 3 mean shift; Sec. 4.1 range of S),
//  * per-point lattice shift m_j = snap(v_j) for the per-point policy (Sec. 4.1, G_{v_j}),
//  * stream compaction of flag arrays into sorted index lists,
//  * marking of the integer domains E_k of the lattice-separable kernel-vector stages,
//  * the reciprocal table w(l) = 1 / (pi^2 (4 l + 2)) (Sec. 3 definition of G_s on the lattice).
#include <float.h>

#include "lsp_internal.h"
#include "snap.cuh"

namespace lsp {
namespace {

constexpr int kThreads = 256;
constexpr int kTileFlags = kThreads * 16;  // flags per compaction tile (one uint4 per thread)

// ---- potential statistics ----
// Minimum and maximum as order-preserving 64-bit integers, reduced by warp instructions on their
// halves; the sum is the only FP64 operation. The FP64 pipe is narrow and its latency long: with
// FP64 shuffles for all four the reductions alone took about 5 us of a launch.
constexpr int kStatThreads = 1024, kStatLoads = 4;

__device__ __forceinline__ unsigned long long order_key(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return b ^ ((unsigned long long)((long long)b >> 63) | (1ULL << 63));
}
__device__ __forceinline__ double key_value(unsigned long long k) {
  return __longlong_as_double((long long)(k ^ (k >> 63 ? 1ULL << 63 : ~0ULL)));
}
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32));
  const unsigned lo =
      __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
  return ((unsigned long long)hi << 32) | lo;
}

struct Stats {
  unsigned long long mn, mx;  // keys
  double sum;
  unsigned bad;  // non-finite values
};
__device__ __forceinline__ Stats empty_stats() {
  return {order_key(DBL_MAX), order_key(-DBL_MAX), 0.0, 0u};
}
__device__ __forceinline__ Stats warp_stats(Stats s) {
  s.mn = ~warp_max_key(~s.mn);
  s.mx = warp_max_key(s.mx);
  s.bad = __reduce_add_sync(0xffffffffu, s.bad);
  for (int o = 16; o > 0; o >>= 1) s.sum += __shfl_xor_sync(0xffffffffu, s.sum, o);
  return s;
}
// Over the block; the result is valid in warp 0.
__device__ __forceinline__ Stats block_stats(Stats s) {
  __shared__ Stats red[kStatThreads / 32];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  s = warp_stats(s);
  if (l == 0) red[w] = s;
  __syncthreads();
  if (w == 0) s = warp_stats(red[l]);  // 32 warps
  return s;
}

// min, max, sum and count of non-finite values of v into out[0..3], and also into host_out[0..3]
// (page-locked host memory, device address) when given, so that the host reads them without a copy.
// With vcopy, v is also stored there (v read from page-locked host memory over the host link, so
// the upload and the statistics take one pass and no copy engine). Every block writes its partial,
// and the block that finishes last (a ticket counter, reset by that block for the next call)
// reduces them, in block order, so the sum does not depend on which block that is.
// Bound by the latency of two reductions; 2^20 points 24 -> 13 us (before: 256 threads a block with
// one load in flight each), 2^10 points 12.7 -> 8.5 us.
__global__ void __launch_bounds__(kStatThreads) k_stats(const double* __restrict__ v, int64_t N,
                                                        Stats* part, double* __restrict__ vcopy,
                                                        double* __restrict__ out,
                                                        double* __restrict__ host_out,
                                                        unsigned int* __restrict__ ticket) {
  Stats s = empty_stats();
  const int64_t step = (int64_t)gridDim.x * kStatThreads;
  for (int64_t j0 = (int64_t)blockIdx.x * kStatThreads + threadIdx.x; j0 < N;
       j0 += kStatLoads * step) {
    double x[kStatLoads];
#pragma unroll
    for (int u = 0; u < kStatLoads; ++u) x[u] = j0 + u * step < N ? v[j0 + u * step] : 0.0;
#pragma unroll
    for (int u = 0; u < kStatLoads; ++u) {
      if (j0 + u * step >= N) break;
      if (vcopy) vcopy[j0 + u * step] = x[u];
      if (((unsigned)__double2hiint(x[u]) & 0x7ff00000u) == 0x7ff00000u) {
        ++s.bad;
        continue;
      }
      const unsigned long long k = order_key(x[u]);
      s.mn = min(s.mn, k);
      s.mx = max(s.mx, k);
      s.sum += x[u];
    }
  }
  s = block_stats(s);
  if (gridDim.x > 1) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
      part[blockIdx.x] = s;
      __threadfence();  // this block's partial is visible before its ticket is taken
      last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    s = threadIdx.x < gridDim.x ? part[threadIdx.x] : empty_stats();
    s = block_stats(s);
    if (threadIdx.x == 0) *ticket = 0u;
  }
  if (threadIdx.x == 0) {
    const double r[4] = {key_value(s.mn), key_value(s.mx), s.sum, (double)s.bad};
    for (int q = 0; q < 4; ++q) out[q] = r[q];
    if (host_out)
      for (int q = 0; q < 4; ++q) host_out[q] = r[q];
  }
}

// The host derived [mlo, mlo + R) from snap(v_min) and snap(v_max) with the same IEEE
// operations; an index outside it would mean the two disagree, and is recorded in *err. Bound by
// the scattered byte stores (2^20 points, 31 us; a look at the flag before the store makes it
// 117 us: the two halves of the L2 pass the written lines back and forth).
__global__ void __launch_bounds__(kThreads) k_mark_local(const double* __restrict__ v, int64_t N,
                                                         int64_t mlo, int64_t R,
                                                         uint8_t* __restrict__ flag,
                                                         int32_t* __restrict__ err) {
  for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < N;
       j += (int64_t)gridDim.x * kThreads) {
    const int64_t r = snap_m(__ldg(v + j)) - mlo;
    if (r >= 0 && r < R)
      flag[r] = 1;
    else
      atomicOr(err, 1);
  }
}

// E_{k-1} gets every l + p^2 for l in the list of E_k and p in [0, P).
__global__ void __launch_bounds__(kThreads) k_mark_stage(const int32_t* __restrict__ list,
                                                         const int32_t* __restrict__ count, int P,
                                                         int64_t lo_prev,
                                                         uint8_t* __restrict__ flag_prev) {
  const int64_t cnt = *count;
  for (int p = blockIdx.y; p < P; p += gridDim.y) {
    const int64_t p2 = (int64_t)p * p;
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < cnt;
         i += (int64_t)gridDim.x * kThreads) {
      flag_prev[(int64_t)__ldg(list + i) + p2 - lo_prev] = 1;
    }
  }
}

__device__ __forceinline__ int count16(uint4 q) {
  return __popc(q.x & 0x01010101u) + __popc(q.y & 0x01010101u) + __popc(q.z & 0x01010101u) +
         __popc(q.w & 0x01010101u);
}

// Compaction pass 1: number of set flags in each tile of kTileFlags.
__global__ void __launch_bounds__(kThreads) k_compact_count(const uint8_t* __restrict__ flag,
                                                            int32_t* __restrict__ tilecnt) {
  const uint4 q = reinterpret_cast<const uint4*>(flag)[(int64_t)blockIdx.x * kThreads + threadIdx.x];
  int c = count16(q);
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  __shared__ int red[kThreads / 32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int w = 0; w < kThreads / 32; ++w) s += red[w];
    tilecnt[blockIdx.x] = s;
  }
}

// Compaction pass 2: exclusive scan of the tile counts (one block), total into *count.
__global__ void __launch_bounds__(1024) k_compact_scan(int32_t* __restrict__ tilecnt, int ntiles,
                                                       int32_t* __restrict__ count) {
  __shared__ int part[1024];
  const int per = (ntiles + 1023) / 1024;
  const int b0 = threadIdx.x * per;
  int s = 0;
  for (int i = 0; i < per; ++i)
    if (b0 + i < ntiles) s += tilecnt[b0 + i];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    int add = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += add;
    __syncthreads();
  }
  int run = part[threadIdx.x] - s;  // exclusive
  for (int i = 0; i < per; ++i) {
    if (b0 + i < ntiles) {
      int c = tilecnt[b0 + i];
      tilecnt[b0 + i] = run;
      run += c;
    }
  }
  if (threadIdx.x == 1023) *count = part[1023];
}

// The list entries of this thread's 16 flags (those of range indices base..), from position pos
// on: list[pos] = lo + r for every set flag r (in increasing r), idx_of[r] = pos (or -1) when
// idx_of is given; with used, the boxes of tree that hold the entry are marked.
__device__ __forceinline__ void write16(uint4 q, int64_t base, int64_t lo, int64_t range, int pos,
                                        int32_t* __restrict__ list, int32_t* __restrict__ idx_of,
                                        const FmmTree& tree, uint8_t* __restrict__ used,
                                        int32_t* __restrict__ err) {
  const uint32_t words[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int64_t r = base + k;
    const bool set = (words[k >> 2] >> (8 * (k & 3))) & 1u;
    if (r < range) {
      if (set) {
        list[pos] = (int32_t)(lo + r);
        if (idx_of) idx_of[r] = pos;
        ++pos;
      } else if (idx_of) {
        idx_of[r] = -1;
      }
    }
  }
  // an aligned group of 16 indices lies in at most two boxes of a level; its set ends mark them
  if (used && (q.x | q.y | q.z | q.w)) {
    int first = 16, last = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if ((words[k >> 2] >> (8 * (k & 3))) & 1u) {
        first = min(first, k);
        last = k;
      }
    if (base + last < range) fmm_mark(tree, lo + base + last, used, err);
    fmm_mark(tree, lo + base + first, used, err);
  }
}

// Inclusive sum of c over the block (at most 32 warps); part holds 32 ints.
__device__ __forceinline__ int block_scan(int c, int* part) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int incl = c;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) part[w] = incl;
  __syncthreads();
  int woff = 0;
  for (int i = 0; i < w; ++i) woff += part[i];
  return woff + incl;
}

// Compaction pass 3: the list entries of every tile.
__global__ void __launch_bounds__(kThreads) k_compact_write(const uint8_t* __restrict__ flag,
                                                            const int32_t* __restrict__ tileoff,
                                                            int64_t lo, int64_t range,
                                                            int32_t* __restrict__ list,
                                                            int32_t* __restrict__ idx_of,
                                                            const __grid_constant__ FmmTree tree,
                                                            uint8_t* __restrict__ used,
                                                            int32_t* __restrict__ err) {
  __shared__ int part[32];
  const int64_t base = (int64_t)blockIdx.x * kTileFlags + (int64_t)threadIdx.x * 16;
  const uint4 q = reinterpret_cast<const uint4*>(flag)[(int64_t)blockIdx.x * kThreads + threadIdx.x];
  const int c = count16(q);
  const int pos = tileoff[blockIdx.x] + block_scan(c, part) - c;
  write16(q, base, lo, range, pos, list, idx_of, tree, used, err);
}

// Up to kOneTiles tiles: the three passes in one launch. Every block counts the flags of all tiles
// before its own (at most 192 KiB, from L2) instead of waiting for a scan. Measured (before: one
// block of 1024 threads): 2D n = 512 (12 tiles) 39 -> 12 us, n = 256 15 -> 10 us; at 72 tiles
// (n = 1024) as long as the three launches.
constexpr int kOneTiles = 48;
__global__ void __launch_bounds__(kThreads) k_compact_one(const uint8_t* __restrict__ flag,
                                                          int64_t lo, int64_t range,
                                                          int32_t* __restrict__ list,
                                                          int32_t* __restrict__ count,
                                                          int32_t* __restrict__ idx_of,
                                                          const __grid_constant__ FmmTree tree,
                                                          uint8_t* __restrict__ used,
                                                          int32_t* __restrict__ err) {
  __shared__ int part[32], before_part[kThreads / 32];
  const uint4* f = reinterpret_cast<const uint4*>(flag);
  const int g = blockIdx.x * kThreads + threadIdx.x;
  const uint4 q = f[g];
  int before = 0;
#pragma unroll 8
  for (int b = 0; b < (int)blockIdx.x; ++b) before += count16(f[b * kThreads + threadIdx.x]);
  before = (int)__reduce_add_sync(0xffffffffu, (unsigned)before);
  if ((threadIdx.x & 31) == 0) before_part[threadIdx.x >> 5] = before;
  const int c = count16(q), incl = block_scan(c, part);  // (its barrier covers before_part)
  before = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) before += before_part[w];
  write16(q, (int64_t)g * 16, lo, range, before + incl - c, list, idx_of, tree, used, err);
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kThreads - 1) *count = before + incl;
}

// w(l) = 1 / (pi^2 (4 l + 2)): FP64 interleaved with w^2, or w alone rounded to FP32.
__global__ void __launch_bounds__(kThreads) k_wtable64(int64_t lo, int64_t range,
                                                       double2* __restrict__ w) {
  for (int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x; r < range;
       r += (int64_t)gridDim.x * kThreads) {
    const double l4 = (double)(4 * (lo + r) + 2);  // exact integer
    const double x = 1.0 / __dmul_rn(kPi2, l4);
    w[r] = make_double2(x, x * x);
  }
}
__global__ void __launch_bounds__(kThreads) k_wtable32(int64_t lo, int64_t range,
                                                       float* __restrict__ w) {
  for (int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x; r < range;
       r += (int64_t)gridDim.x * kThreads) {
    const double l4 = (double)(4 * (lo + r) + 2);
    w[r] = (float)(1.0 / __dmul_rn(kPi2, l4));
  }
}

// Double words (hi, lo floats) of w and w^2 from their FP64 values, interleaved per l.
__global__ void __launch_bounds__(kThreads) k_wtable_dw(int64_t lo, int64_t range,
                                                        float4* __restrict__ w) {
  for (int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x; r < range;
       r += (int64_t)gridDim.x * kThreads) {
    const double l4 = (double)(4 * (lo + r) + 2);
    const double x = 1.0 / __dmul_rn(kPi2, l4), x2 = x * x;
    const float xh = (float)x, x2h = (float)x2;
    w[r] = make_float4(xh, (float)(x - (double)xh), x2h, (float)(x2 - (double)x2h));
  }
}

int grid_for(int64_t work, int per_block = kThreads) {
  int64_t b = (work + per_block - 1) / per_block;
  const int64_t cap = 152 * 32;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (int)b;
}

// Zeroes n 32-bit words. A kernel rather than a memset, so that the build never waits behind
// host copies queued on the copy engines.
__global__ void __launch_bounds__(kThreads) k_zero_u32(uint32_t* __restrict__ p, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * kThreads)
    p[i] = 0u;
}

__global__ void __launch_bounds__(kThreads) k_zero3_u32(uint32_t* __restrict__ a, int64_t na,
                                                        uint32_t* __restrict__ b, int64_t nb,
                                                        uint32_t* __restrict__ d, int64_t nd) {
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < na + nb + nd;
       i += (int64_t)gridDim.x * kThreads) {
    if (i < na)
      a[i] = 0u;
    else if (i < na + nb)
      b[i - na] = 0u;
    else
      d[i - na - nb] = 0u;
  }
}

// dst[0, n) = src[0, n) (doubles; both 16-byte aligned): pairs by every thread, an odd last
// element by thread 0.
__global__ void __launch_bounds__(kThreads) k_copy_f64(const double* __restrict__ src,
                                                       double* __restrict__ dst, int64_t n) {
  const int64_t n2 = n / 2;
  const double2* s2 = reinterpret_cast<const double2*>(src);
  double2* d2 = reinterpret_cast<double2*>(dst);
  const int64_t t0 = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  for (int64_t i = t0; i < n2; i += (int64_t)gridDim.x * kThreads) d2[i] = s2[i];
  if (t0 == 0 && (n & 1)) dst[n - 1] = src[n - 1];
}

}  // namespace

// One load of every thread in flight per block and SM, and a single block (no ticket) for small grids.
int stats_blocks(int64_t N) {
  const int64_t b = (N + kStatThreads * kStatLoads - 1) / (kStatThreads * kStatLoads);
  return (int)(b < 152 ? b : 152);
}
size_t stats_part_bytes(int64_t N) { return sizeof(Stats) * stats_blocks(N); }

cudaError_t launch_stats(lsp_ctx* c, const double* src) {
  int t = timer_begin(c, "stats");
  double* vd = (double*)c->v.p;
  double* st = (double*)c->stats.p;
  k_stats<<<stats_blocks(c->geo.N), kStatThreads, 0, c->stream>>>(
      src, c->geo.N, (Stats*)c->stats_part.p, src == vd ? nullptr : vd, st, c->h_stats_dev,
      (unsigned int*)(st + 4));
  timer_end(c, t);
  return cudaGetLastError();
}

cudaError_t launch_zero(lsp_ctx* c, void* p, size_t bytes) {
  const int64_t n = (int64_t)(bytes / 4);
  int t = timer_begin(c, "zero");
  k_zero_u32<<<grid_for(n), kThreads, 0, c->stream>>>((uint32_t*)p, n);
  timer_end(c, t);
  return cudaGetLastError();
}

cudaError_t launch_zero3(lsp_ctx* c, ZeroRange a, ZeroRange b, ZeroRange d) {
  const int64_t na = (int64_t)(a.bytes / 4), nb = (int64_t)(b.bytes / 4);
  const int64_t nd = (int64_t)(d.bytes / 4);
  int t = timer_begin(c, "zero");
  k_zero3_u32<<<grid_for(na + nb + nd), kThreads, 0, c->stream>>>(
      (uint32_t*)a.p, na, (uint32_t*)b.p, nb, (uint32_t*)d.p, nd);
  timer_end(c, t);
  return cudaGetLastError();
}

cudaError_t launch_copy_f64(lsp_ctx* c, const double* src, double* dst, int64_t n) {
  int t = timer_begin(c, "copy_rows");
  k_copy_f64<<<grid_for((n + 1) / 2), kThreads, 0, c->stream>>>(src, dst, n);
  timer_end(c, t);
  return cudaGetLastError();
}

cudaError_t launch_mark_local(lsp_ctx* c) {
  int t = timer_begin(c, "mark_local");
  k_mark_local<<<grid_for(c->geo.N), kThreads, 0, c->stream>>>(
      (const double*)c->v.p, c->geo.N, c->mrange.lo, c->mrange.size(), (uint8_t*)c->shift_flag.p,
      (int32_t*)c->counts.p + kErrWord);
  timer_end(c, t);
  return cudaGetLastError();
}

// flags must hold a multiple of kTileFlags bytes (zero beyond `range`); tile scratch lives in
// the context's `counts` buffer after its first 16 entries.
cudaError_t launch_compact(lsp_ctx* c, const uint8_t* flags, int64_t lo, int64_t range,
                           int32_t* list, int32_t* count, int32_t* idx_of, const FmmTree* tree,
                           uint8_t* used) {
  int32_t* err = (int32_t*)c->counts.p + kErrWord;
  const FmmTree t = tree ? *tree : FmmTree{};
  if (!tree) used = nullptr;
  const int ntiles = (int)((range + kTileFlags - 1) / kTileFlags);
  int32_t* tiles = (int32_t*)c->counts.p + 16;
  int tm = timer_begin(c, "compact");
  if (ntiles <= kOneTiles) {
    k_compact_one<<<ntiles, kThreads, 0, c->stream>>>(flags, lo, range, list, count, idx_of, t,
                                                      used, err);
  } else {
    k_compact_count<<<ntiles, kThreads, 0, c->stream>>>(flags, tiles);
    k_compact_scan<<<1, 1024, 0, c->stream>>>(tiles, ntiles, count);
    k_compact_write<<<ntiles, kThreads, 0, c->stream>>>(flags, tiles, lo, range, list, idx_of, t,
                                                        used, err);
  }
  timer_end(c, tm);
  return cudaGetLastError();
}

cudaError_t launch_mark_stage(lsp_ctx* c, const int32_t* list, const int32_t* count, int64_t cap,
                              int64_t lo_prev, uint8_t* flag_prev) {
  const int P = c->geo.P;
  int gx = (int)((cap + kThreads - 1) / kThreads);
  if (gx > 1024) gx = 1024;
  if (gx < 1) gx = 1;
  dim3 grid(gx, P < 4096 ? P : 4096);
  int t = timer_begin(c, "mark_stage");
  k_mark_stage<<<grid, kThreads, 0, c->stream>>>(list, count, P, lo_prev, flag_prev);
  timer_end(c, t);
  return cudaGetLastError();
}

cudaError_t launch_wtable(lsp_ctx* c, int64_t lo, int64_t range, void* w, int prec) {
  int t = timer_begin(c, "wtable");
  if (prec == kPrecFP32)
    k_wtable32<<<grid_for(range), kThreads, 0, c->stream>>>(lo, range, (float*)w);
  else if (prec == kPrecDword)
    k_wtable_dw<<<grid_for(range), kThreads, 0, c->stream>>>(lo, range, (float4*)w);
  else
    k_wtable64<<<grid_for(range), kThreads, 0, c->stream>>>(lo, range, (double2*)w);
  timer_end(c, t);
  return cudaGetLastError();
}

}  // namespace lsp
