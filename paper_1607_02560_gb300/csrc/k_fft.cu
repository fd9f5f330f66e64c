// y = (L + diag(v)) u with L = F^-1 diag(4 pi^2 |k|^2) F (Sec. 2, Eq. dmodel).
//
// |k|^2 is a sum over the axes and F a tensor product, so L = sum_a D_a with D_a the 1D operator
// F_1^-1 diag(4 pi^2 k_a^2) F_1 along axis a. Each D_a maps real lines to real lines, so two lines
// travel through one complex transform as its real and imaginary parts: half the operations of
// a complex transform of the whole grid, no complex array in memory, and one pass per axis:
//   last axis: t = D u;  middle axis (3D): t += D u;  axis 0 (1D: the only one): y = D u + t + v u.
//
// What bounds it: the FP64 pipe (2 lanes per SM per clock). A complex value costs 66 FP64
// instructions an axis at n = 1024, i.e. 110 us for the million points of 2D n = 1024; the
// bytes (48 a point) would take 7 us and stay in L2. A block transforms W pairs of lines in shared memory,
// in place: forward passes with decreasing spans leave the spectrum in digit-reversed order, the
// innermost pass applies the symbol between its forward and inverse butterflies in registers,
// and the inverse passes retrace the spans, so no reordering is needed. Passes of radix 4: as
// many operations as radix 8 and more threads per line. The kernels of one call overlap: a later
// axis' blocks start as the earlier ones drain and wait only before they read t and store, which
// also hides their launch (2D n = 64 21 -> 14 us, n = 1024 172 -> 147 us).
// Measured against complex transforms of the whole grid in radix-2 passes: 2D n = 1024 418 ->
// 147 us (0.75 of the FP64 rate), n = 64 29 -> 14 us, 3D n = 64 125 -> 37 us, 1D n = 1024
// 39 -> 25 us; the error against extended precision is smaller (random u 0.5 to 0.9 of it, smooth
// packets 0.6 to 0.95 over 1D n = 64 to 4096, 2D 16 to 512 and 3D 8, 32; 2D n = 16 with plane waves
// equal).
#include <type_traits>

#include "lsp_internal.h"

namespace lsp {
namespace {

// Twiddle table of an axis length n: tw[j] = exp(-2 pi i j / n), j < n, then sym[k] =
// 4 pi^2 min(k, n - k)^2 / n, k < n (the 1/n of the inverse transform, exact, folded in).
struct AxisTable {
  const double2* tw;
  const double* sym;
};
AxisTable axis_table(const double* p, int n) {
  return {reinterpret_cast<const double2*>(p), p + 2 * (size_t)n};
}

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
// a * w (or a * conj(w) for the inverse)
template <bool INV>
__device__ __forceinline__ double2 ctw(double2 a, double2 w) {
  return INV ? make_double2(fma(a.x, w.x, a.y * w.y), fma(a.y, w.x, -(a.x * w.y)))
             : make_double2(fma(a.x, w.x, -(a.y * w.y)), fma(a.x, w.y, a.y * w.x));
}
// -i a (forward) or i a (inverse)
template <bool INV>
__device__ __forceinline__ double2 rot(double2 a) {
  return INV ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x);
}

template <bool INV>
__device__ __forceinline__ void dft4(double2& a, double2& b, double2& c, double2& d) {
  const double2 s0 = cadd(a, c), d0 = csub(a, c), s1 = cadd(b, d), r = rot<INV>(csub(b, d));
  a = cadd(s0, s1);
  c = csub(s0, s1);
  b = cadd(d0, r);
  d = csub(d0, r);
}
template <int R, bool INV>
__device__ __forceinline__ void dft(double2 (&x)[R]) {
  if constexpr (R == 4) {
    dft4<INV>(x[0], x[1], x[2], x[3]);
  } else {
    constexpr double c = 0.70710678118654752440;  // cos(pi / 4)
    dft4<INV>(x[0], x[2], x[4], x[6]);  // even inputs: E_0..E_3
    dft4<INV>(x[1], x[3], x[5], x[7]);  // odd inputs: O_0..O_3
    const double2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    const double2 o0 = x[1], o2 = rot<INV>(x[5]);
    // O_1 w and O_3 w^3 without their factor cos(pi / 4)
    const double2 o1 = INV ? make_double2(x[3].x - x[3].y, x[3].x + x[3].y)
                           : make_double2(x[3].x + x[3].y, x[3].y - x[3].x);
    const double2 o3 = INV ? make_double2(-(x[7].x + x[7].y), x[7].x - x[7].y)
                           : make_double2(x[7].y - x[7].x, -(x[7].x + x[7].y));
    x[0] = cadd(e0, o0);
    x[4] = csub(e0, o0);
    x[2] = cadd(e2, o2);
    x[6] = csub(e2, o2);
    x[1] = make_double2(fma(c, o1.x, e1.x), fma(c, o1.y, e1.y));
    x[5] = make_double2(fma(-c, o1.x, e1.x), fma(-c, o1.y, e1.y));
    x[3] = make_double2(fma(c, o3.x, e3.x), fma(c, o3.y, e3.y));
    x[7] = make_double2(fma(-c, o3.x, e3.x), fma(-c, o3.y, e3.y));
  }
}

// Radix plan of n = 2^LOGN: one pass of 8 where LOGN is odd, then passes of 4.
template <int LOGN>
struct Plan {
  static constexpr int n = 1 << LOGN;
  static constexpr int passes = LOGN / 2;
  __host__ __device__ static constexpr int radix(int s) { return LOGN % 2 && s == 0 ? 8 : 4; }
  __host__ __device__ static constexpr int span(int s) {  // length of the sub-transforms of pass s
    int L = n;
    for (int i = 0; i < s; ++i) L /= radix(i);
    return L;
  }
};
static_assert(Plan<3>::passes == 1 && Plan<4>::passes == 2 && Plan<12>::passes == 6, "plan");

// Shared-memory place of element i of a line: one element of padding per 8 keeps the strided
// accesses of every pass free of bank conflicts.
__host__ __device__ constexpr int padded(int i) { return i + (i >> 3); }
template <int LOGN>
__host__ __device__ constexpr int line_slots() {  // per line; = 2 (mod 8) so that lines spread over banks
  return ((padded((1 << LOGN) - 1) + 1 + 5) / 8) * 8 + 2;
}

struct LineArgs {
  const double* u;    // input
  const double* t;    // sum of the axes already done (null for the first)
  const double* v;    // potential: final pass only (null otherwise)
  double* out;        // may be u in the final pass: each thread reads u[g] before it writes out[g]
  int64_t stride;     // between the elements of a line: 1 (last axis) or n, n^2
  int64_t npairs;     // pairs of lines (1D: one line, its partner is zero)
  int single;         // 1D
  int wlog;           // log2 of the pairs per block
  int vec;            // u, t, v, out may be accessed as 16-byte pairs (strided axes)
  AxisTable tab;
};

// One axis. STRIDED: pairs are neighbours along the last axis, (u[g], u[g + 1]) is one complex
// value, and a block's W pairs are consecutive, so a row of the block is 16 W bytes. Otherwise
// pairs are consecutive lines. Work items of a pass: (pair, j) with j the position inside the
// pass's span; W = 2^wlog pairs share a block.
template <int LOGN, bool STRIDED>
__global__ void __launch_bounds__(256) k_axis(LineArgs a) {
  using P = Plan<LOGN>;
  constexpr int n = P::n, SLOTS = line_slots<LOGN>();
  extern __shared__ double2 sm[];
  // The next axis' blocks may start: they read u, and wait (below) before they touch t or y.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int W = 1 << a.wlog;
  const int64_t pair0 = (int64_t)blockIdx.x << a.wlog;
  // address of element 0 of pair q of this block
  auto base_of = [&](int q) -> int64_t {
    const int64_t pr = pair0 + q;
    if (!STRIDED) return pr * 2 * n;  // lines 2 pr and 2 pr + 1
    const int64_t half = a.stride >> 1, outer = pr / half;
    return outer * a.stride * n + 2 * (pr - outer * half);
  };
  auto load = [&](int64_t b, int i) -> double2 {
    if (STRIDED) {
      const int64_t g = b + (int64_t)i * a.stride;
      if (a.vec) return *reinterpret_cast<const double2*>(a.u + g);
      return make_double2(a.u[g], a.u[g + 1]);
    }
    return make_double2(a.u[b + i], a.single ? 0.0 : a.u[b + n + i]);
  };
  auto store = [&](int64_t b, int i, double2 z) {
    const int64_t g0 = STRIDED ? b + (int64_t)i * a.stride : b + i;
    const int64_t g1 = STRIDED ? g0 + 1 : g0 + n;
    if (STRIDED && a.vec) {
      if (a.t) {
        const double2 t = *reinterpret_cast<const double2*>(a.t + g0);
        z = cadd(z, t);
      }
      if (a.v) {
        const double2 u = *reinterpret_cast<const double2*>(a.u + g0);
        const double2 v = *reinterpret_cast<const double2*>(a.v + g0);
        z = make_double2(fma(v.x, u.x, z.x), fma(v.y, u.y, z.y));
      }
      *reinterpret_cast<double2*>(a.out + g0) = z;
      return;
    }
    if (a.t) z.x += a.t[g0];
    if (a.v) z.x = fma(a.v[g0], a.u[g0], z.x);
    if (a.single) {
      a.out[g0] = z.x;
      return;
    }
    if (a.t) z.y += a.t[g1];
    if (a.v) z.y = fma(a.v[g1], a.u[g1], z.y);
    a.out[g0] = z.x;
    a.out[g1] = z.y;
  };
  // Before the first store of a later axis: the previous axis' kernel has completed, so t is
  // whole, and y may overwrite u.
  auto previous_axis = [&]() {
    if (a.t) asm volatile("griddepcontrol.wait;" ::: "memory");
  };
  // item e -> (pair, position j in [0, n / R))
  auto item = [&](int e, int per, int& q, int& j) {
    if (STRIDED) {
      q = e & (W - 1);
      j = e >> a.wlog;
    } else {
      q = e / per;
      j = e - q * per;
    }
  };
  auto run = [&](auto self, auto sc) -> void {
    constexpr int s = decltype(sc)::value;
    constexpr int R = P::radix(s), L = P::span(s), QS = L / R, per = n / R;
    constexpr bool first = s == 0, last = s == P::passes - 1;
    // forward: x_r = in[b + j + r QS]; X_f *= w_L^{j f}; back in place
    for (int e = threadIdx.x; e < (per << a.wlog); e += blockDim.x) {
      int q, p;
      item(e, per, q, p);
      const int blk = p / QS, j = p - blk * QS, i0 = blk * L + j;
      double2* line = sm + q * SLOTS;
      double2 x[R];
      if (first) {
        const int64_t b = base_of(q);
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = load(b, i0 + r * QS);
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = line[padded(i0 + r * QS)];
      }
      dft<R, false>(x);
      if constexpr (!last) {
#pragma unroll
        for (int f = 1; f < R; ++f) x[f] = ctw<false>(x[f], __ldg(a.tab.tw + (n / L) * j * f));
#pragma unroll
        for (int r = 0; r < R; ++r) line[padded(i0 + r * QS)] = x[r];
      } else {
        // QS = 1: outputs are the frequencies k0 + (n / R) f, k0 the reversed digits of blk
        int k0 = 0, rem = i0;
#pragma unroll
        for (int d = 0; d < s; ++d) {
          const int q2 = P::span(d + 1), dig = rem / q2;
          rem -= dig * q2;
          k0 += dig * (n / P::span(d));
        }
#pragma unroll
        for (int f = 0; f < R; ++f) {
          const double lam = __ldg(a.tab.sym + k0 + (n / R) * f);
          x[f].x *= lam;
          x[f].y *= lam;
        }
        dft<R, true>(x);
        if (first) {  // a single pass (n = 8): straight out
          previous_axis();
          const int64_t b = base_of(q);
#pragma unroll
          for (int r = 0; r < R; ++r) store(b, i0 + r * QS, x[r]);
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) line[padded(i0 + r * QS)] = x[r];
        }
      }
    }
    if constexpr (!last) {
      __syncthreads();
      self(self, std::integral_constant<int, s + 1>{});
      // inverse: x_f = in * conj(w_L^{j f}); inverse butterflies; back in place (or out)
      if (first) previous_axis();
      for (int e = threadIdx.x; e < (per << a.wlog); e += blockDim.x) {
        int q, p;
        item(e, per, q, p);
        const int blk = p / QS, j = p - blk * QS, i0 = blk * L + j;
        double2* line = sm + q * SLOTS;
        double2 x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = line[padded(i0 + r * QS)];
#pragma unroll
        for (int f = 1; f < R; ++f) x[f] = ctw<true>(x[f], __ldg(a.tab.tw + (n / L) * j * f));
        dft<R, true>(x);
        if (first) {
          const int64_t b = base_of(q);
#pragma unroll
          for (int r = 0; r < R; ++r) store(b, i0 + r * QS, x[r]);
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) line[padded(i0 + r * QS)] = x[r];
        }
      }
      if constexpr (!first) __syncthreads();
    } else if constexpr (!first) {
      __syncthreads();
    }
  };
  run(run, std::integral_constant<int, 0>{});
}

template <int LOGN>
cudaError_t launch_axis_n(LineArgs a, cudaStream_t st) {
  const bool strided = a.stride > 1;
  // Pairs per block: enough work items (n / 4 a pair) for a whole warp, since a partly filled
  // warp costs the FP64 pipe as much as a full one (3D n = 64 with one pair: 78 us against 37),
  // and two on strided axes with pairs enough for 16 blocks per SM, where rows of 32 bytes pay
  // (3D n = 128 416 -> 327 us). With fewer, single pairs spread more evenly over the SMs (2D
  // n = 1024 264 -> 147 us, the second axis' blocks joining the first's; 2D n = 256 20 -> 16 us).
  const size_t line = sizeof(double2) * line_slots<LOGN>();
  const int64_t rows = strided ? a.stride / 2 : a.npairs;  // the pairs per block divide this
  a.wlog = 0;
  while (rows % (2 << a.wlog) == 0 &&
         ((Plan<LOGN>::n << a.wlog) < 128 ||
          (strided && a.wlog == 0 && LOGN <= 10 && a.npairs >= 16 * 152)))
    ++a.wlog;
  const size_t smem = Plan<LOGN>::passes > 1 ? line << a.wlog : 0;
  const int items = (Plan<LOGN>::n / 4) << a.wlog;
  const int threads = items < 32 ? 32 : (items > 256 ? 256 : items);
  const int64_t blocks = a.npairs >> a.wlog;
  auto go = [&](auto kern) -> cudaError_t {
    if (smem > 48 * 1024) {
      cudaError_t e =
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = a.t ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, a);
  };
  return strided ? go(k_axis<LOGN, true>) : go(k_axis<LOGN, false>);
}

// y = (L + diag v) u on the n^d grid; t: n^d doubles of scratch (d > 1), tab: the axis table.
cudaError_t apply_axes(int d, int n, const double* u, const double* v, double* y, double* t,
                       const double* tab, cudaStream_t st) {
  int logn = 0;
  while ((1 << logn) < n) ++logn;
  int64_t N = 1, S = 1;
  for (int i = 0; i < d; ++i) N *= n;
  for (int axis = d - 1; axis >= 0; --axis, S *= n) {
    LineArgs a;
    a.u = u;
    a.t = axis < d - 1 ? t : nullptr;
    a.v = axis == 0 ? v : nullptr;
    a.out = axis == 0 ? y : t;
    a.stride = S;
    a.single = d == 1;
    a.npairs = d == 1 ? 1 : N / n / 2;
    a.wlog = 0;
    a.vec = (((uintptr_t)u | (uintptr_t)v | (uintptr_t)y | (uintptr_t)t) & 15) == 0;
    a.tab = axis_table(tab, n);
    cudaError_t e = cudaErrorInvalidValue;
    switch (logn) {
      case 3: e = launch_axis_n<3>(a, st); break;
      case 4: e = launch_axis_n<4>(a, st); break;
      case 5: e = launch_axis_n<5>(a, st); break;
      case 6: e = launch_axis_n<6>(a, st); break;
      case 7: e = launch_axis_n<7>(a, st); break;
      case 8: e = launch_axis_n<8>(a, st); break;
      case 9: e = launch_axis_n<9>(a, st); break;
      case 10: e = launch_axis_n<10>(a, st); break;
      case 11: e = launch_axis_n<11>(a, st); break;
      case 12: e = launch_axis_n<12>(a, st); break;
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_apply(lsp_ctx* c, const double* u, double* y) {
  int t = timer_begin(c, "apply_fft");
  cudaError_t e = apply_axes(c->geo.d, c->geo.n, u, (const double*)c->v.p, y,
                             (double*)c->fftbuf.p, (const double*)c->twiddle.p, c->stream);
  timer_end(c, t);
  return e;
}

}  // namespace lsp

// ---- y = (L + diag v) u without any device allocation -------------------------------------
// Some callers cannot allocate device memory at the moment they need the operator: code that
// runs while a CUDA stream is being captured into a graph (where cudaMalloc is not permitted),
// and code whose device memory is owned by a pool or framework allocator that forbids extra
// allocations, or that cannot afford the device-wide synchronisation a cudaMalloc may cause.
// For them the scratch of the transform lives in a fixed, file-scope device array instead of a
// context buffer. Every GPU that loads this library holds that array (8 MiB of scratch plus
// 24 KiB of tables) until the process exits.
namespace lsp {
namespace {

constexpr int64_t kNoAllocMaxPoints = (int64_t)1 << 20;  // must match LSP_NOALLOC_MAX_POINTS
constexpr int kNoAllocMaxN = 1024;  // d >= 2 and n^d <= 2^20
static __device__ __align__(256) double g_noalloc_work[kNoAllocMaxPoints];
static __device__ __align__(256) double g_noalloc_table[3 * kNoAllocMaxN];

// The axis table (see AxisTable) with the CUDA math library's sincospi.
__global__ void k_noalloc_table(double* __restrict__ tab, int n) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    double s, c;
    sincospi(2.0 * (double)j / (double)n, &s, &c);
    tab[2 * j] = c;
    tab[2 * j + 1] = -s;
    const double k = j < n / 2 ? (double)j : (double)(j - n);
    tab[2 * n + j] = 4.0 * kPi2 * (k * k) / (double)n;
  }
}

}  // namespace
}  // namespace lsp

extern "C" lsp_status lsp_apply_operator_noalloc(int d, int n, const double* v_dev,
                                                 const double* u_dev, double* y_dev,
                                                 void* cuda_stream) {
  using namespace lsp;
  if (d != 2 && d != 3) return LSP_ERR_ARG;
  if (n < 8 || (n & (n - 1)) != 0 || n > 2 * 2048) return LSP_ERR_ARG;
  int64_t N = 1;
  for (int i = 0; i < d; ++i) N *= n;
  if (N > kNoAllocMaxPoints) return LSP_ERR_ARG;  // larger grids need the context path
  if (!v_dev || !u_dev || !y_dev) return LSP_ERR_ARG;
  // The symbol names are host-side stand-ins, not device addresses, so they are never passed
  // to a kernel. Their device addresses are looked up on every call, in the current device's
  // current context: the lookup allocates nothing, and a cached address could outlive a
  // context that was torn down and created again. The first call in a context loads the
  // library's device code there, so make it before any stream capture.
  double* work = nullptr;
  double* tab = nullptr;
  if (cudaGetSymbolAddress((void**)&work, g_noalloc_work) != cudaSuccess ||
      cudaGetSymbolAddress((void**)&tab, g_noalloc_table) != cudaSuccess) {
    cudaGetLastError();
    return LSP_ERR_CUDA;
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  cudaGetLastError();
  k_noalloc_table<<<(n + 255) / 256, 256, 0, st>>>(tab, n);
  // the first pass writes every element of the scratch before any pass reads it, so it needs
  // no clearing between calls
  return apply_axes(d, n, u_dev, v_dev, y_dev, work, tab, st) == cudaSuccess ? LSP_OK
                                                                             : LSP_ERR_CUDA;
}
