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


@pytest.mark.parametrize("d,n,leaf", [(2, 64, 32), (3, 16, 8)])
@pytest.mark.parametrize("kind", ["blocks", "log"])
def test_rows_of_very_different_scales(d, n, leaf, kind):
    """One listed shift for a potential of nine (blocks of rows) to eleven (every row) orders of
    magnitude: rows of P up to 1e5 times larger than others inside one step of 64 pivots, whose
    digits are taken relative to the largest entry of a row or column. Each row by itself: the plain
    solve contracts (1e-7) and one refinement step leaves the rounding of a residual of mu products,
    (mu + 2) u of sum |P| |x| + |y|."""
    rng = np.random.default_rng(n)
    N = n ** d
    s0 = 18 * O.PI2
    f, sign = rng.random((n,) * d), rng.choice([-1.0, 1.0], (n,) * d)
    if kind == "log":
        v = s0 + 10.0 ** (11 * f - 3) * sign
    else:
        v = np.where(np.indices((n,) * d)[0] % 7 < 2, 1e9 * (0.5 + 0.5 * f), s0 + 100 * f * sign)
    ctx = ctx_for(v)
    ctx.set_potential(v)
    ctx.build_stencils(policy="list", shifts=np.array([s0]))
    P = csr(ctx, "P", N)
    rows = abs(P).max(axis=1).toarray()
    assert rows.max() > 1e3 * rows.min()
    y = P @ rng.standard_normal(N)
    for steps, tol in ((0, 1e-7), (1, (3 ** d + 2) * U)):
        ctx.nd_factor(leaf=leaf, refine_steps=steps)
        x = gpu_solve(ctx, y)
        err = np.abs(P @ x - y) / (abs(P) @ np.abs(x) + np.abs(y))
        assert err.max() <= tol, (steps, err.max())
