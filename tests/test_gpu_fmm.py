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


@pytest.mark.parametrize("more", [0, 1300, 40000])
@pytest.mark.parametrize("d,n", [(2, 128), (2, 256), (3, 64)])
def test_kernel_vectors_as_accurate_as_direct_sums(d, n, more):
    """c = G alpha with the returned alpha and G summed in extended precision, for shifts across the
    range of a potential; more consecutive shifts in the list bring the kernels for longer lists.
    Unit: 2^-53 of the shift's largest g. Sums over the frequencies axis by axis leave G's entries
    about 1 unit off in 2D and 1/3 in 3D (rms), and the product with the unit vector alpha adds 1/2
    (2D) and 2/3 (3D): at most 1.5 and 1 together."""
    import itertools
    import torch
    from paper_1607_02560_gb300 import Context
    R = np.longdouble
    v = make_workload("helm2d_n256" if d == 2 else "schr3d_n64", n=n)
    ms = np.unique(np.round((v.ravel() / PI2 - 2.0) / 4.0).astype(int))
    ms = ms[np.linspace(0, len(ms) - 1, min(len(ms), 60)).astype(int)]
    every = np.union1d(ms, np.arange(ms[0], ms[0] + more))
    ctx = Context(d, n, stream=torch.cuda.Stream())
    ctx.set_potential(v)
    ctx.build_stencils(policy="list", shifts=(4.0 * every + 2.0) * PI2)
    t = ctx.get_shift_table(with_sidx=False)
    at = np.searchsorted(every, ms)
    alpha, c = t["alpha"][at].astype(R), t["c"][at].astype(R)
    two_pi = 8 * np.arctan(R(1))
    p = np.arange(n // 2 + 1)
    wgt = np.where((p == 0) | (p == n // 2), R(1), R(2))
    X = np.stack([wgt * np.cos(two_pi * ((a * p) % n).astype(R) / n) for a in range(3)])
    r = sum((p * p).reshape([-1 if a == b else 1 for b in range(d)]) for a in range(d))
    offs = np.array(list(itertools.product((-1, 0, 1), repeat=d)))
    diff = tuple(np.moveaxis(np.abs(offs[:, None] - offs[None]), -1, 0))
    off = []
    for i, m in enumerate(ms):
        g = 1 / (R(PI2) * (4 * (r + int(m)) + 2).astype(R))
        for _ in range(d):
            g = np.tensordot(g, X, axes=([0], [1]))
        g = g / R(n) ** d
        off.append((c[i] - g[diff] @ alpha[i]) / (np.abs(g).max() * R(2) ** -53))
    rms = float(np.sqrt(np.mean(np.array(off, dtype=float) ** 2)))
    assert rms <= (1.5 if d == 2 else 1.0), rms
