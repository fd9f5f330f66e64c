"""The blocked partial inversion at the edges of its steps: fronts just above the size swept in
shared memory, a last step of one pivot, a last panel of one pivot, several panels per row of
threads, and panels of more than 2048 rows, against the sparse LU of the same P."""

import numpy as np
import pytest

import oracle as O
from lsp_inputs import make_workload
from test_gpu_nd import U, backward_error, csr, ctx_for, gpu_solve, kappa_1

pytestmark = pytest.mark.gpu


# leaf fronts: 225 + 64 (225 = 3 * 64 + 2 * 16 + 1), 961 + 124 (961 = 15 * 64 + 1), 343 + 169
# (343 = 5 * 64 + 23), 3375 + 721 (3375 = 52 * 64 + 47 rows: the panel with its rows in memory)
@pytest.mark.parametrize("d,n,leaf", [(2, 64, 16), (2, 32, 32), (3, 8, 8), (3, 16, 16)])
def test_step_remainders(d, n, leaf):
    """One refinement step leaves the rounding of a residual of at most 27 products (backward
    error below 1e-15 of 9 max|P| max|x| + max|y|) and the forward error of a backward stable solve
    (256 u kappa). The plain solve contracts (1e-7 as at full size: pivots are chosen inside a
    front); a second factorisation gives the same bits."""
    v = make_workload("helm2d_n32" if d == 2 else "schr3d_n64", n=n)
    N = n ** d
    ctx = ctx_for(v)
    ctx.set_potential(v)
    ctx.build_stencils(policy="local")
    P = csr(ctx, "P", N)
    y = np.random.default_rng(n + leaf).standard_normal(N)
    ctx.nd_factor(leaf=leaf)
    plain = gpu_solve(ctx, y)
    ctx.nd_factor(leaf=leaf)
    assert np.array_equal(gpu_solve(ctx, y), plain)
    assert backward_error(P, plain, y) <= 1e-7
    ctx.nd_factor(leaf=leaf, refine_steps=1)
    x = gpu_solve(ctx, y)
    assert backward_error(P, x, y) <= 1e-15
    ref = O.solve_p(P, y)
    assert np.abs(x - ref).max() <= 256 * U * kappa_1(P) * np.abs(ref).max()
