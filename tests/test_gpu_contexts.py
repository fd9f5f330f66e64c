"""Several contexts alive at once: what one of them sets up is not seen by the others."""

import numpy as np
import pytest

from lsp_inputs import make_workload

pytestmark = pytest.mark.gpu

GRIDS = {1: ("helm1d_n256", 64), 2: ("helm2d_n32", 32), 3: ("schr3d_n64", 16)}


def context(d, n=None):
    import torch
    from paper_1607_02560_gb300 import Context
    name, n0 = GRIDS[d]
    ctx = Context(d, n or n0, stream=torch.cuda.Stream())
    ctx.set_potential(make_workload(name, n=n or n0))
    return ctx


def rows(ctx, **kw):
    ctx.build_stencils(policy="local", **kw)
    return [ctx.get_rows(w) for w in "QCP"] + [ctx.get_shift_table(with_sidx=False)["lam"]]


@pytest.mark.parametrize("kw", [{}, dict(eig_method="full"), dict(refine_steps=1)])
def test_dimensions_do_not_share_tables(kw):
    """The first build of each dimension, made before the others exist, is repeated bit for bit
    after contexts of the other dimensions were made, in every order."""
    first = {}
    for d in (2, 3, 1):
        ctx = context(d)
        first[d] = rows(ctx, **kw)
        ctx.close()
    for order in ((1, 2, 3), (3, 2, 1), (2, 3, 1), (3, 1, 2)):
        ctxs = {d: context(d) for d in order}
        for d in order:
            for a, b in zip(rows(ctxs[d], **kw), first[d]):
                assert np.array_equal(a, b), (order, d)


def test_a_smaller_plan_leaves_a_larger_solve_alone():
    """A plan of small fronts, made by another context after a plan of large ones: the large
    solve (9 to 24 KiB of shared memory more than the small one's) gives the same bits, and both
    factorise again."""
    import torch
    large, small = context(2, 512), context(2, 16)
    for ctx in (large, small):
        ctx.build_stencils(policy="paper")
    y = torch.from_numpy(np.random.default_rng(0).standard_normal(512 * 512)).cuda()
    x, x2 = torch.empty_like(y), torch.empty_like(y)
    torch.cuda.synchronize()
    large.nd_factor(leaf=8)
    large.nd_solve(y, x)
    large.synchronize()
    small.nd_factor(leaf=8)
    large.nd_solve(y, x2)
    large.synchronize()
    assert torch.equal(x, x2)
    large.nd_factor(leaf=8)
    large.nd_solve(y, x2)
    large.synchronize()
    assert torch.equal(x, x2)
