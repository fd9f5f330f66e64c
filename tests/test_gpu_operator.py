"""The pseudospectral operator at every axis length and layout it is dispatched on, against a
transform of the whole grid."""

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n", [(1, 8), (1, 16), (1, 32), (1, 128), (1, 4096), (2, 8), (2, 16),
                                 (2, 32), (2, 512), (2, 2048), (3, 8), (3, 16), (3, 32), (3, 128)])
@pytest.mark.parametrize("shift", [0, 1])
def test_operator_sizes_and_alignment(d, n, shift):
    """shift = 1: u and y start 8 bytes past a 16-byte boundary (scalar accesses on strided axes).

    Tolerance: the transforms' rounding, a few units per pass relative to the largest symbol, as
    in the other operator tests (1e-13 of the operator's norm times max |u|)."""
    import torch
    from paper_1607_02560_gb300 import Context
    rng = np.random.default_rng(n + d)
    shape = (n,) * d
    v = -(2 * np.pi * n / 4) ** 2 * rng.uniform(0.5, 1.5, shape)
    u = rng.standard_normal(shape)
    stream = torch.cuda.Stream()
    ctx = Context(d, n, stream=stream)
    ctx.set_potential(v)
    ub = torch.zeros(n ** d + 1, dtype=torch.float64, device="cuda")
    yb = torch.full_like(ub, np.nan)
    ub[shift:shift + n ** d] = torch.from_numpy(u.reshape(-1)).cuda()
    uw, yw = ub[shift:shift + n ** d], yb[shift:shift + n ** d]
    torch.cuda.synchronize()
    ref = O.apply_operator(v, u).reshape(-1)
    tol = 1e-13 * (4 * O.PI2 * d * (n / 2) ** 2 + np.abs(v).max()) * np.abs(u).max()
    ctx.apply_operator(uw, yw)
    ctx.synchronize()
    assert np.abs(yw.cpu().numpy() - ref).max() <= tol
    first = yw.clone()
    ctx.apply_operator(uw, uw)  # in place: the same operations on the same values
    ctx.synchronize()
    assert torch.equal(uw, first)
    assert float(ub[n ** d if shift == 0 else 0]) == 0.0  # nothing outside the array


@pytest.mark.parametrize("d,n", [(2, 64), (3, 16)])
def test_noalloc_operator_in_a_captured_graph(d, n):
    """The overlapping kernels of one call keep their order inside a CUDA graph: replays on new
    inputs equal the context's call."""
    import torch
    from paper_1607_02560_gb300 import Context, lsp
    rng = np.random.default_rng(1)
    v = torch.from_numpy(-1e4 * rng.uniform(0.5, 1.5, (n,) * d)).cuda()
    u, y, ref = torch.zeros_like(v), torch.zeros_like(v), torch.zeros_like(v)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = Context(d, n, stream=stream)
    ctx.set_potential(v)
    lsp.apply_operator_noalloc(d, n, v, u, y, stream=stream)  # loads the library's device code
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for _ in range(3):  # y = A^3 u, in place after the first
            lsp.apply_operator_noalloc(d, n, v, u if _ == 0 else y, y, stream=stream)
    for seed in range(2):
        u.copy_(torch.from_numpy(np.random.default_rng(seed).standard_normal((n,) * d)).cuda())
        torch.cuda.synchronize()
        g.replay()
        for k in range(3):
            ctx.apply_operator(u if k == 0 else ref, ref)
        ctx.synchronize()
        torch.cuda.synchronize()
        assert float((y - ref).abs().max()) <= 1e-12 * float(ref.abs().max())
