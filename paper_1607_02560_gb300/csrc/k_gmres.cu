// Device side of restarted GMRES (Sec. 5: restart 40, relative tolerance 1e-6) for
// (L + diag v) u = f, left-preconditioned by P^-1 C (Eq. PC). The Arnoldi basis V, the
// Hessenberg matrix H (column-major, leading dimension ld = restart + 1), the Givens rotations
// and the least-squares right-hand side S all stay on the device; the host loop reads back one
// residual estimate per inner iteration. Reductions use a fixed grid and a fixed summation
// order, so two runs on the same data take the same decisions.
#include <math.h>

#include "nd.h"

namespace lsp {
namespace {

constexpr int kRedBlocks = 1024;  // <= the partial-sum slots of GmresSlot
constexpr int kRedThreads = 256;

int red_grid(int64_t N) {
  const int64_t b = (N + kRedThreads - 1) / kRedThreads;
  return (int)(b < kRedBlocks ? (b > 0 ? b : 1) : kRedBlocks);
}

// w -= h_prev * v_prev (when v_prev), then *h_out = sum_i v_next[i] w[i] (or w[i]^2).
// The last block to finish adds the block partials in block order.
__global__ void __launch_bounds__(kRedThreads) k_mgs(double* w,
                                                     const double* __restrict__ v_prev,
                                                     const double* h_prev,
                                                     const double* __restrict__ v_next,
                                                     double* gs, double* h_out, int64_t N) {
  __shared__ double wsum[kRedThreads / 32];
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // Launched to overlap the kernel before: the basis vectors were complete before that one
  // started, so their first values are on the way while it finishes.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NP = 4;
  const int64_t i0 = blockIdx.x * (int64_t)kRedThreads + tid, step = (int64_t)gridDim.x * kRedThreads;
  double vp[NP], vn[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    const int64_t i = i0 + k * step;
    vp[k] = v_prev && i < N ? __ldg(v_prev + i) : 0.0;
    vn[k] = v_next && i < N ? __ldg(v_next + i) : 0.0;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const double h = v_prev ? *h_prev : 0.0;
  double acc = 0.0;
  for (int64_t ib = i0; ib < N; ib += NP * step) {
    double wv[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) wv[k] = ib + k * step < N ? w[ib + k * step] : 0.0;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int64_t i = ib + k * step;
      if (i >= N) break;
      double wi = wv[k];
      if (v_prev) {
        wi = fma(-h, vp[k], wi);
        w[i] = wi;
      }
      acc = fma(v_next ? vn[k] : wi, wi, acc);
    }
    const int64_t nx = ib + NP * step;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int64_t i = nx + k * step;
      vp[k] = v_prev && i < N ? __ldg(v_prev + i) : 0.0;
      vn[k] = v_next && i < N ? __ldg(v_next + i) : 0.0;
    }
  }
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (lane == 0) wsum[warp] = acc;
  __syncthreads();
  if (tid == 0) {
    double b = 0.0;
    for (int k = 0; k < kRedThreads / 32; ++k) b += wsum[k];
    gs[kGsPartial + blockIdx.x] = b;
    __threadfence();
    const unsigned t = atomicAdd((unsigned*)(gs + kGsTicket), 1u);
    last = t == gridDim.x - 1;
  }
  __syncthreads();
  if (last && warp == 0) {
    __threadfence();
    double b = 0.0;
    for (int k = lane; k < (int)gridDim.x; k += 32) b += __ldcg(gs + kGsPartial + k);
    for (int off = 16; off > 0; off >>= 1) b += __shfl_xor_sync(0xffffffffu, b, off);
    if (lane == 0) {
      *h_out = b;
      *(unsigned*)(gs + kGsTicket) = 0u;
    }
  }
}

// y[i] = (a ? a[i] : 0) + sign * (scale ? *scale : 1) * x[i]
__global__ void k_axpby(double* __restrict__ y, const double* a, const double* x,
                        const double* __restrict__ scale, double sign, int64_t N) {
  const double sc = sign * (scale ? *scale : 1.0);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = fma(sc, x[i], a ? a[i] : 0.0);
}

// v0 = r / beta with beta = sqrt(gs[kGsNorm]); S = (beta, 0, ...).
__global__ void k_gmres_start(double* __restrict__ gs, int ld, int restart,
                              const double* __restrict__ r, double* __restrict__ v0, int64_t N) {
  __shared__ double sinv;
  const double beta = sqrt(gs[kGsNorm]);
  if (threadIdx.x == 0) sinv = beta > 0.0 ? 1.0 / beta : 0.0;  // one division per block
  __syncthreads();
  const double inv = sinv;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x)
    v0[i] = r[i] * inv;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    double* S = gs + kGsArrays + (int64_t)ld * restart + 2 * restart;
    for (int k = 0; k < ld; ++k) S[k] = 0.0;
    S[0] = beta;
    gs[kGsBeta] = beta;
  }
}

// Column col of H holds <v_k, w> (k <= col) from the MGS steps; complete it with |w|, apply
// the previous rotations, make the rotation that zeroes H[col + 1][col], rotate S.
__device__ void givens_column(double* gs, int col, int ld, int restart) {
  double* H = gs + kGsArrays;
  double* cs = H + (int64_t)ld * restart;
  double* sn = cs + restart;
  double* S = sn + restart;
  double* hc = H + (int64_t)col * ld;
  const double h0 = sqrt(gs[kGsH0]), h1 = sqrt(gs[kGsH1]);
  const bool brk = !(h1 > 2.220446049250313e-16 * h0);
  gs[kGsBreak] = brk ? 1.0 : 0.0;
  gs[kGsInvH1] = brk ? 0.0 : 1.0 / h1;
  hc[col + 1] = brk ? 0.0 : h1;
  for (int k = 0; k < col; ++k) {
    const double a = hc[k], b = hc[k + 1];
    hc[k] = cs[k] * a + sn[k] * b;
    hc[k + 1] = -sn[k] * a + cs[k] * b;
  }
  const double a = hc[col], b = hc[col + 1];
  const double rr = hypot(a, b);
  double c = 1.0, s = 0.0;
  if (rr > 0.0) {
    c = a / rr;
    s = b / rr;
  }
  cs[col] = c;
  sn[col] = s;
  hc[col] = rr;
  hc[col + 1] = 0.0;
  S[col + 1] = -s * S[col];
  S[col] = c * S[col];
  gs[kGsPresid] = fabs(S[col + 1]);
}

__global__ void k_gmres_givens(double* gs, int col, int ld, int restart) {
  if (blockIdx.x == 0 && threadIdx.x == 0) givens_column(gs, col, ld, restart);
}

// One Arnoldi column: modified Gram-Schmidt of w against v_0..v_col, |w| before and after, the
// Givens rotations, v_{col+1} = w / |w|. Cooperative: every block keeps its part of w in
// registers from the first projection to the last, so a projection reads v_k once (and the next
// one while the blocks exchange their partial sums) instead of w twice and v_k twice, and the
// blocks meet once per projection instead of ending a kernel. Bound by the FP64 pipe (2 N
// products a projection, 3.3 us at N = 2^20) and the meeting (about 2 us): 9.1 us a projection, where
// one kernel each took 14.4 us and the gap to the next launch. Every block adds all partial sums in
// block order, so all have the same h and the result is deterministic. The wait for the others is bounded (1 s); when it
// runs out, gs[kGsFail] is set and every block leaves.
constexpr int kArnThreads = 1024, kArnPer = 8;
__device__ __forceinline__ bool meet(unsigned* bar, unsigned target, bool ok) {
  __shared__ bool s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    uint64_t t0 = 0;
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if ((int)(v - target) >= 0 || !ok) break;
      uint64_t t;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
      if (t0 == 0) t0 = t;
      if (t - t0 > 1000000000ull) {
        ok = false;
        break;
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok;
}

// Sum of x over the block, in every thread's return value of warp 0 (fixed order).
__device__ __forceinline__ double block_sum(double x, double* sh) {
  const int tid = threadIdx.x;
  __syncthreads();
  sh[tid] = x;
  __syncthreads();
  if (tid < 128) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += sh[tid + 128 * k];
    sh[tid] = s;
  }
  __syncthreads();
  double s = 0.0;
  if (tid < 32) {
    s = (sh[tid] + sh[tid + 32]) + (sh[tid + 64] + sh[tid + 96]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  return s;
}

__global__ void __launch_bounds__(kArnThreads, 1) k_arnoldi(const double* __restrict__ w,
                                                            double* V, double* gs, int col, int ld,
                                                            int restart, int64_t N, unsigned* bar,
                                                            unsigned base) {
  __shared__ double sh[kArnThreads];
  __shared__ double s_h, s_h0;
  const int tid = threadIdx.x, G = gridDim.x;
  const int64_t per = (N + G - 1) / G, lo = blockIdx.x * per;
  const int64_t hi = lo + per < N ? lo + per : N;
  double wv[kArnPer], vv[kArnPer];
#pragma unroll
  for (int e = 0; e < kArnPer; ++e) {
    const int64_t i = lo + tid + e * kArnThreads;
    wv[e] = i < hi ? w[i] : 0.0;
    vv[e] = i < hi ? V[i] : 0.0;
  }
  double* hc = gs + kGsArrays + (int64_t)col * ld;
  bool ok = true;
  // all partial sums of one exchange, added in block order by warp 0 of every block
  auto total = [&](const double* p) {
    double s = 0.0;
    for (int b = tid; b < G; b += 32) s += __ldcg(p + b);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  for (int k = 0; k <= col + 1 && ok; ++k) {
    // exchange k: <v_k, w> (k <= col), |w|^2 after the last projection; the first also |w|^2
    double* p = gs + kGsPartial + (k & 1) * 512;
    double acc = 0.0, acc0 = 0.0;
#pragma unroll
    for (int e = 0; e < kArnPer; ++e) acc = fma(k <= col ? vv[e] : wv[e], wv[e], acc);
    const double bs = block_sum(acc, sh);
    if (tid == 0) p[blockIdx.x] = bs;
    if (k == 0) {
#pragma unroll
      for (int e = 0; e < kArnPer; ++e) acc0 = fma(wv[e], wv[e], acc0);
      const double b0 = block_sum(acc0, sh);
      if (tid == 0) p[256 + blockIdx.x] = b0;
    }
    double vn[kArnPer];
    if (k < col) {  // the next basis vector arrives while the blocks meet
      const double* v = V + (int64_t)(k + 1) * N;
#pragma unroll
      for (int e = 0; e < kArnPer; ++e) {
        const int64_t i = lo + tid + e * kArnThreads;
        vn[e] = i < hi ? v[i] : 0.0;
      }
    }
    ok = meet(bar, base + (unsigned)(k + 1) * G, ok);
    if (!ok) break;
    if (tid < 32) {
      const double h = total(p);
      const double h0 = k == 0 ? total(p + 256) : 0.0;
      if (tid == 0) {
        s_h = h;
        if (k == 0) s_h0 = h0;
        if (blockIdx.x == 0 && k <= col) hc[k] = h;
      }
    }
    __syncthreads();
    const double h = s_h;
    if (k <= col) {
#pragma unroll
      for (int e = 0; e < kArnPer; ++e) {
        wv[e] = fma(-h, vv[e], wv[e]);
        vv[e] = k < col ? vn[e] : 0.0;
      }
    }
    __syncthreads();  // s_h is read before the next exchange writes it
  }
  if (!ok) {
    if (tid == 0) gs[kGsFail] = 1.0;
    return;
  }
  // s_h: |w|^2 after; the same decision as givens_column
  const double h0 = sqrt(s_h0), h1 = sqrt(s_h);
  if (tid == 0) sh[0] = !(h1 > 2.220446049250313e-16 * h0) ? 0.0 : 1.0 / h1;
  if (blockIdx.x == 0 && tid == 0) {
    gs[kGsH0] = s_h0;
    gs[kGsH1] = s_h;
    givens_column(gs, col, ld, restart);
  }
  __syncthreads();
  const double inv = sh[0];
  double* vo = V + (int64_t)(col + 1) * N;
#pragma unroll
  for (int e = 0; e < kArnPer; ++e) {
    const int64_t i = lo + tid + e * kArnThreads;
    if (i < hi) vo[i] = wv[e] * inv;
  }
}

// y = H[0..col, 0..col]^-1 S[0..col] (back substitution, in every block), x += V[:, 0..col] y.
__global__ void k_gmres_update(const double* __restrict__ gs, int col, int ld, int restart,
                               const double* __restrict__ V, double* __restrict__ x, int64_t N) {
  __shared__ double y[64];
  if (threadIdx.x == 0) {
    const double* H = gs + kGsArrays;
    const double* S = H + (int64_t)ld * restart + 2 * restart;
    for (int k = col; k >= 0; --k) {
      double v = S[k];
      for (int j = k + 1; j <= col; ++j) v -= H[(int64_t)j * ld + k] * y[j];
      const double d = H[(int64_t)k * ld + k];
      y[k] = d != 0.0 ? v / d : 0.0;
    }
  }
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x) {
    double acc = x[i];
    for (int k = 0; k <= col; ++k) acc = fma(y[k], V[(int64_t)k * N + i], acc);
    x[i] = acc;
  }
}

int ew_grid(int64_t N) {
  const int64_t b = (N + 255) / 256;
  return (int)(b < 152 * 8 ? (b > 0 ? b : 1) : 152 * 8);
}

}  // namespace

cudaError_t launch_mgs(lsp_ctx* c, double* w, const double* v_prev, const double* h_prev,
                       const double* v_next, double* h_out, int64_t N) {
  double* gs = (double*)c->nd->gs.p;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(red_grid(N));
  cfg.blockDim = dim3(kRedThreads);
  cfg.stream = c->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mgs, w, v_prev, h_prev, v_next, gs, h_out, N);
}

bool arnoldi_fits(lsp_ctx* c, int64_t N) {
  NdState& S = *c->nd;
  if (S.coop_blocks < 0) {
    int sms = 0, per = 0, coop = 0;
    S.coop_blocks = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) == cudaSuccess &&
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, c->device) == cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_arnoldi, kArnThreads, 0) ==
            cudaSuccess &&
        coop && per > 0)
      S.coop_blocks = sms < 256 ? sms : 256;  // partial-sum slots
    cudaGetLastError();
  }
  return S.coop_blocks > 0 && N <= (int64_t)S.coop_blocks * kArnThreads * kArnPer;
}

cudaError_t launch_arnoldi(lsp_ctx* c, const double* w, double* V, double* gs, int col, int ld,
                           int64_t N) {
  NdState& S = *c->nd;
  int64_t G = (N + kArnThreads - 1) / kArnThreads;
  if (G > S.coop_blocks) G = S.coop_blocks;
  unsigned* bar = (unsigned*)S.bar.p;
  unsigned base = S.bar_count;
  int restart = ld - 1;
  void* args[] = {&w, &V, &gs, &col, &ld, &restart, &N, &bar, &base};
  const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_arnoldi, dim3((unsigned)G),
                                                    dim3(kArnThreads), args, 0, c->stream);
  if (e == cudaSuccess) S.bar_count += (unsigned)G * (unsigned)(col + 2);
  return e;
}

cudaError_t launch_axpby(lsp_ctx* c, double* y, const double* a, const double* x,
                         const double* scale, double sign, int64_t N) {
  k_axpby<<<ew_grid(N), 256, 0, c->stream>>>(y, a, x, scale, sign, N);
  return cudaGetLastError();
}

cudaError_t launch_gmres_start(lsp_ctx* c, double* gs, int ld, const double* r, double* v0,
                               int64_t N) {
  k_gmres_start<<<ew_grid(N), 256, 0, c->stream>>>(gs, ld, ld - 1, r, v0, N);
  return cudaGetLastError();
}

cudaError_t launch_gmres_givens(lsp_ctx* c, double* gs, int col, int ld) {
  k_gmres_givens<<<1, 32, 0, c->stream>>>(gs, col, ld, ld - 1);
  return cudaGetLastError();
}

cudaError_t launch_gmres_update(lsp_ctx* c, double* gs, int col, int ld, const double* V,
                                double* x, int64_t N) {
  k_gmres_update<<<ew_grid(N), 256, 0, c->stream>>>(gs, col, ld, ld - 1, V, x, N);
  return cudaGetLastError();
}

}  // namespace lsp
