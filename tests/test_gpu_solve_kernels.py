"""The kernels of the Krylov solve at the edges of their dispatch: the row products for every row
width, and the Arnoldi column in one launch (grids up to about 1.2 million points) or one kernel
per projection (larger), against plain numpy."""

import numpy as np
import pytest
import scipy.sparse

import oracle as O
from lsp_inputs import make_workload

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def context(d, n, v):
    import torch
    from paper_1607_02560_gb300 import Context
    ctx = Context(d, n, stream=torch.cuda.Stream())
    ctx.set_potential(v)
    return ctx


@pytest.mark.parametrize("d,n,t", [(1, 8, 1), (1, 256, 1), (2, 8, 1), (2, 64, 1), (2, 16, 2),
                                   (3, 8, 1), (3, 16, 1), (3, 16, 2)])
def test_row_products_for_every_row_width(d, n, t):
    """Fewer points than a block, whole blocks, 3 to 125 entries a row. Tolerance: a row's FMA
    chain of mu <= 125 terms, mu u times the sum of their magnitudes (512 u covers it)."""
    import torch
    name = {1: "helm1d_n256", 2: "helm2d_n256", 3: "schr3d_n64"}[d]
    ctx = context(d, n, make_workload(name, n=n))
    ctx.build_stencils(policy="paper", t=t, nd_leaf=8 if t == 2 else 0)
    N = n ** d
    u = np.random.default_rng(n).standard_normal(N)
    ud = torch.from_numpy(u).cuda()
    yd = torch.empty_like(ud)
    torch.cuda.synchronize()
    for which in "QCP":
        rowptr, colidx, vals = ctx.export_sparse_rows(which)
        M = scipy.sparse.csr_matrix((vals, colidx, rowptr), shape=(N, N))
        ctx.apply_rows(which, ud, yd)
        ctx.synchronize()
        err = np.abs(yd.cpu().numpy() - M @ u)
        assert (err <= 512 * U * (abs(M) @ np.abs(u))).all(), which


def gmres_numpy(v, f, steps):
    """`steps` steps of GMRES with modified Gram-Schmidt, no preconditioner, x0 = 0."""
    V = [f.ravel() / np.linalg.norm(f)]
    H = np.zeros((steps + 1, steps))
    for k in range(steps):
        w = O.apply_operator(v, V[k].reshape(v.shape)).ravel()
        for i in range(k + 1):
            H[i, k] = V[i] @ w
            w = w - H[i, k] * V[i]
        H[k + 1, k] = np.linalg.norm(w)
        V.append(w / H[k + 1, k])
    e = np.zeros(steps + 1)
    e[0] = np.linalg.norm(f)
    y = np.linalg.lstsq(H, e, rcond=None)[0]
    return sum(c * b for c, b in zip(y, V)), np.linalg.norm(e - H @ y) / e[0]


@pytest.mark.parametrize("d,n,steps", [(1, 8, 5), (1, 4096, 1), (2, 64, 2), (2, 1024, 1),
                                       (2, 2048, 1), (3, 32, 1)])
def test_arnoldi_columns(d, n, steps):
    """One block, one block per SM with an uneven share, and more points than the registers of
    one launch hold. Without the preconditioner every application turns rounding of size u into
    high frequencies and multiplies it by the largest eigenvalue, 4 pi^2 d (n/2)^2, against the
    smallest, v >= 400: tolerance 64 u (their ratio)^steps, at least 1e-11."""
    x = np.arange(n) / n
    ax = [x.reshape([n if a == b else 1 for b in range(d)]) for a in range(d)]
    one = np.ones((n,) * d)
    v = np.ascontiguousarray(sum(400.0 * (2 + np.cos(2 * np.pi * (a + 0.1))) for a in ax) * one)
    f = np.ascontiguousarray(sum(np.cos(2 * np.pi * (k + 1) * a) for k, a in enumerate(ax)) * one)
    tol = max(1e-11, 64 * U * (4 * O.PI2 * d * (n / 2) ** 2 / 400.0 + 3 * d) ** steps)
    ctx = context(d, n, v)
    u, res = ctx.gmres(f.ravel(), rtol=1e-30, restart=steps, max_cycles=1, precond=False)
    ref, rel = gmres_numpy(v, f, steps)
    assert res["iterations"] == steps and res["converged"] == 0
    assert np.abs(u - ref).max() <= tol * np.abs(ref).max()
    assert abs(res["resid_true"] - rel) <= max(tol, 1e-9)
    u2, _ = ctx.gmres(f.ravel(), rtol=1e-30, restart=steps, max_cycles=1, precond=False)
    assert np.array_equal(u, u2)


@pytest.mark.parametrize("n,leaf", [(1024, 4), (256, 4)])
def test_more_fronts_than_a_second_grid_dimension_holds(n, leaf):
    """The smallest leaves of the largest grid: 65 536 fronts at one depth. One refinement step
    leaves the rounding of a residual of nine products: backward error below 1e-15 of
    9 max|P| max|x| + max|y|."""
    import torch
    ctx = context(2, n, make_workload("helm2d_n256", n=n))
    ctx.build_stencils(policy="paper")
    ctx.nd_factor(leaf=leaf, refine_steps=1)
    y = torch.from_numpy(np.random.default_rng(n).standard_normal(n * n)).cuda()
    x, r = torch.empty_like(y), torch.empty_like(y)
    torch.cuda.synchronize()
    ctx.nd_solve(y, x)
    ctx.apply_rows("P", x, r)
    rows = ctx.get_rows("P")
    scale = 9 * np.abs(rows).max() * x.abs().max().item() + y.abs().max().item()
    assert (r - y).abs().max().item() <= 1e-15 * scale
