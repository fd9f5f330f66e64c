"""Device functions that stand in for FP64 arithmetic, on their own: the pivots' reciprocal against
CUDA's correctly rounded division, the digits of the error-free split and the sum of its levels
against exact integers."""

import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <stdint.h>
#include "recip.cuh"
#include "digits.cuh"
__global__ void k_recip(const double* x, double* r, double* q, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    r[i] = lsp::recip_f64(x[i]);
    q[i] = 1.0 / x[i];
  }
}
__global__ void k_digits(const double* x, const int* e, int* d, int* ex, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    int v[lsp::kDigits];
    lsp::digits_of(x[i], e[i], v);
    for (int t = 0; t < lsp::kDigits; ++t) d[i * lsp::kDigits + t] = v[t];
    ex[i] = lsp::exp_of(x[i]);
  }
}
__global__ void k_sum(const int* a, const int* ex, double* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    int v[lsp::kLevels];
    for (int l = 0; l < lsp::kLevels; ++l) v[l] = a[i * lsp::kLevels + l];
    s[i] = lsp::sum_of(v, ex[i]);
  }
}
extern "C" int run(int which, const void* a, const void* b, void* c, void* d, int n) {
  const int g = (n + 255) / 256;
  if (which == 0) k_recip<<<g, 256>>>((const double*)a, (double*)c, (double*)d, n);
  if (which == 1) k_digits<<<g, 256>>>((const double*)a, (const int*)b, (int*)c, (int*)d, n);
  if (which == 2) k_sum<<<g, 256>>>((const int*)a, (const int*)b, (double*)c, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    from paper_1607_02560_gb300 import build
    tmp = tmp_path_factory.mktemp("device")
    src, lib = tmp / "f.cu", tmp / "f.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o",
                    str(lib), str(src)], check=True, capture_output=True)
    fn = ctypes.CDLL(str(lib)).run

    def call(which, a, b, *outs):
        dev = [torch.from_numpy(np.ascontiguousarray(t)).cuda() for t in (a, b, *outs)]
        torch.cuda.synchronize()
        ptr = [ctypes.c_void_p(t.data_ptr()) for t in dev] + [None] * (4 - len(dev))
        assert fn(which, *ptr, len(a)) == 0
        return [t.cpu().numpy() for t in dev[2:]]

    return call


def patterns(rng, n):
    """Doubles of every exponent, with random mantissas and with mantissas next to powers of two."""
    mant = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    edge = rng.integers(0, 3, n)
    near = rng.integers(0, 4, n).astype(np.uint64)
    mant = np.where(edge == 1, near, np.where(edge == 2, np.uint64((1 << 52) - 1) - near, mant))
    expo = rng.integers(0, 2048, n).astype(np.uint64)
    sign = rng.integers(0, 2, n).astype(np.uint64)
    return ((sign << np.uint64(63)) | (expo << np.uint64(52)) | mant).view(np.float64)


def test_reciprocal_of_a_pivot(run):
    """Less than 0.51 ulp off the exact value, so at most one representable number away from the
    correctly rounded division (and mostly the same); zeros, subnormals, infinities, NaN and results
    that are not normal are the division's."""
    x = patterns(np.random.default_rng(0), 1 << 20)
    x[:8] = [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.0 ** -1022, 1.7976931348623157e308]
    r, q = run(0, x, x, np.empty_like(x), np.empty_like(x))
    normal = np.isfinite(x) & (np.abs(x) >= 2.0 ** -1022) & (np.abs(q) >= 2.0 ** -1022) \
        & np.isfinite(q)
    assert np.array_equal(r[~normal].view(np.int64)[~np.isnan(r[~normal])],
                          q[~normal].view(np.int64)[~np.isnan(q[~normal])])
    apart = np.abs(r[normal].view(np.int64) - q[normal].view(np.int64))
    assert apart.max() <= 1
    some = np.flatnonzero(normal)[:20000]
    for i in some[apart[:20000] > 0]:
        exact = 1 / Fraction(x[i])
        ulp = Fraction(float(np.spacing(np.abs(r[i]))))
        assert abs(Fraction(r[i]) - exact) < Fraction(51, 100) * ulp


def test_digits_of_values_far_below_the_largest(run):
    """x = sum of d[t] 512^(6 - t) 2^(e - 62), rounded to that unit once, for values down to 2^-70 of
    2^e; balanced digits, so every product of two fits an FP32 sum of 64 exactly."""
    rng = np.random.default_rng(1)
    n = 20000
    x = rng.uniform(0.5, 1.0, n) * rng.choice([-1.0, 1.0], n)
    x[::7] = rng.choice([0.5, -0.5, 1.0 - 2.0 ** -53, 2.0 ** -53 - 1.0], len(x[::7]))
    e = rng.integers(-900, 900, n).astype(np.int32)
    drop = rng.integers(0, 71, n)
    x = np.ldexp(x, e - drop)
    x[::11] = 0.0
    d, ex = run(1, x, e, np.empty((n, 7), np.int32), np.empty(n, np.int32))
    assert np.abs(d).max() <= 256 and d[:, 1:].max() <= 255
    zero = x == 0.0
    assert (ex[~zero] == np.frexp(x[~zero])[1]).all() and (ex[zero] < -99999).all()
    for i in range(0, n, 5):
        value = sum(int(d[i, t]) * 512 ** (6 - t) for t in range(7))
        exact = Fraction(x[i]) * Fraction(2) ** (62 - int(e[i]))
        assert abs(value - exact) <= Fraction(1, 2)
        if drop[i] <= 9:
            assert value == exact


def test_sum_of_levels_is_rounded_once(run):
    """sum a[l] 2^(ex - 9 l) for |a[l]| <= 2^24, from levels of one size to levels that cancel: half
    an ulp and the 2^-11 ulp of what lies below its leading 64 bits; zero below the normal range and
    infinite above it."""
    rng = np.random.default_rng(2)
    n = 20000
    size = rng.integers(0, 25, (n, 7))
    a = (rng.integers(-1, 2, (n, 7)) * (np.int64(1) << size)
         + rng.integers(-3, 4, (n, 7))).clip(-(1 << 24), 1 << 24)
    a[::3, 0] = 0
    a[::9, :4] = 0
    k = np.arange(0, n, 10)  # leading levels that cancel but for a small rest
    a[k, 1] = rng.integers(-(1 << 14), 1 << 14, len(k))
    a[k, 0] = 0
    a[k, 2] = -512 * a[k, 1]
    a[5] = 0
    ex = rng.integers(-900, 900, n).astype(np.int32)
    ex[1::50] = rng.integers(-1100, -1020, len(ex[1::50]))
    ex[2::50] = rng.integers(990, 1030, len(ex[2::50]))
    s, = run(2, a.astype(np.int32), ex, np.empty(n))
    low, high = Fraction(2) ** -1022, Fraction(2) ** 1024
    for i in range(n):
        exact = sum(Fraction(int(a[i, l]), 512 ** l) for l in range(7)) * Fraction(2) ** int(ex[i])
        if abs(exact) < low * (1 - Fraction(1, 1 << 50)):
            assert s[i] == 0.0
        elif abs(exact) >= high:
            assert np.isinf(s[i]) and (s[i] > 0) == (exact > 0)
        elif low * 2 < abs(exact) < high / 2:
            ulp = Fraction(float(np.spacing(np.abs(s[i]))))
            assert abs(Fraction(s[i]) - exact) <= (Fraction(1, 2) + Fraction(1, 2048)) * ulp, i
