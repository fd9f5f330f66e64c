"""The fast multipole evaluation of the kernel vectors (t = 1, FP64, 2D and 3D) against the
stage-by-stage sums, which t = 2 builds use for all their stencils: with nd_leaf = 8 the points
next to a separator carry the t = 1 stencil of their shift in the inner columns of the row.

Tolerances: alpha moves by u kappa_gap under a rounding-level change of the kernel vectors (2D
kappa_gap <= 250, 3D <= 2.5e6; 16 such changes allowed): 2D 1e-11 covers 250 * 16 * 2^-53 =
4e-13 with the longer sums' rounding, 3D 5e-9 is 2.5e6 * 16 * 2^-53. The C entries follow alpha
through |G| alpha, relative to the largest one."""

import numpy as np
import pytest

from lsp_inputs import make_workload

pytestmark = pytest.mark.gpu

PI2 = np.pi * np.pi


def points_with_narrow_rows(d, n, leaf=8):
    r = np.arange(n) % leaf
    f = np.where(r == 0, leaf, np.minimum(r, leaf - r))
    t = np.minimum(2, f)
    full = t.reshape([n] + [1] * (d - 1))
    for a in range(1, d):
        full = np.minimum(full, t.reshape([n if a == b else 1 for b in range(d)]))
    return np.flatnonzero(full.reshape(-1) == 1)


def compare(d, n, v, **kw):
    import torch
    from paper_1607_02560_gb300 import Context
    ctx = Context(d, n, stream=torch.cuda.Stream())
    ctx.set_potential(v)
    ctx.build_stencils(t=1, **kw)
    one = {w: ctx.get_rows(w) for w in "QC"}
    ctx.build_stencils(t=2, nd_leaf=8, **kw)
    two = {w: ctx.get_rows(w) for w in "QC"}
    offs = np.stack(np.meshgrid(*([np.arange(-2, 3)] * d), indexing="ij"), -1).reshape(-1, d)
    inner = np.flatnonzero((np.abs(offs) <= 1).all(1))
    pts = points_with_narrow_rows(d, n)
    tol = 1e-11 if d == 2 else 5e-9
    for w in "QC":
        a, b = one[w][pts], two[w][pts][:, inner]
        assert np.abs(a - b).max() <= tol * np.abs(b).max(), (w, np.abs(a - b).max())
    assert np.array_equal(one["Q"][pts[0]] > 0, two["Q"][pts[0]][inner] > 0)


@pytest.mark.parametrize("d,n,policy", [(2, 8, "local"), (2, 32, "local"), (2, 64, "paper"),
                                        (2, 128, "local"), (2, 256, "paper"), (2, 512, "local"),
                                        (3, 8, "local"), (3, 16, "paper"), (3, 32, "local")])
def test_multipole_sums_equal_the_stages(d, n, policy):
    """One block, eight lanes and two lanes per shift; trees of one to a dozen levels."""
    compare(d, n, make_workload("helm2d_n256" if d == 2 else "schr3d_n64", n=n), policy=policy)


@pytest.mark.parametrize("d,n", [(2, 16), (2, 64), (3, 16)])
def test_shifts_beyond_the_frequencies_and_at_box_edges(d, n):
    """Listed shifts on both sides of zero and of -|p|^2_max, at and around multiples of the box
    width 128, and a single one, against the oracle with the parity tests' per-shift tolerance
    max(1e-10, 16 u kappa_gap)."""
    import torch
    from paper_1607_02560_gb300 import Context
    from test_gpu_parity import check_shift_table
    top = d * (n // 2) ** 2
    edges = [-128 * k + e for k in (0, 1, 2, 4, top // 128) for e in (-1, 0, 1)]
    m = sorted(set(edges + [-2 * top, -top - 200, -top, -top // 2, -7, 3, 127, 128, 300]))
    rng = np.random.default_rng(n)
    pick = rng.choice(len(m), n ** d)
    pick[:len(m)] = np.arange(len(m))
    shifts = (4.0 * np.array(m) + 2.0) * PI2
    v = shifts[pick].reshape((n,) * d)
    ctx = Context(d, n, stream=torch.cuda.Stream())
    ctx.set_potential(v)
    for part in (m, m[:1]):
        ctx.build_stencils(policy="list", shifts=shifts[:len(part)])
        check_shift_table(ctx.get_shift_table(), v, "list", m_list=part)


@pytest.mark.parametrize("d,n", [(2, 8), (2, 64), (3, 16)])
def test_shifts_up_to_the_largest_index(d, n):
    """Listed shifts far beyond the frequencies, up to the largest lattice index a build takes.
    There the sums are almost w(m) times the identity: G has the eigenvalues w(m + r) of a
    projection of functions of |p|^2 = r <= r_max, so |G - w(m)| <= w(m) r_max / (|m| - r_max) in the
    spectral norm, and |c - w(m) alpha| is at most that for the unit vector alpha. (alpha itself is
    not determined to any digit.) Rounding: at most 1e-12 of w(m)."""
    import torch
    from paper_1607_02560_gb300 import Context
    r_max = d * (n // 2) ** 2
    ctx = Context(d, n, stream=torch.cuda.Stream())
    ctx.set_potential(make_workload("helm2d_n256" if d == 2 else "schr3d_n64", n=n))
    big = 2147483000 - 4 * r_max
    for ms in ((2 ** 29 + 5,), (2 ** 30 - 1, 2 ** 30, 2 ** 30 + 1, 2 ** 30 + 300), (1100000000,),
               (big - 200, big), (-2 ** 30 - 1, -2 ** 30), (-big,)):
        shifts = (4.0 * np.array(ms) + 2.0) * PI2
        ctx.build_stencils(policy="list", shifts=shifts)
        t = ctx.get_shift_table(with_sidx=False)
        assert len(t["s"]) == len(ms)
        for m, s, alpha, c in zip(ms, t["s"], t["alpha"], t["c"]):
            assert abs(np.linalg.norm(alpha) - 1.0) <= 1e-12, m
            tol = r_max / (abs(m) - r_max) + 1e-12
            assert np.linalg.norm(c * s - alpha) <= tol, (m, np.linalg.norm(c * s - alpha))
