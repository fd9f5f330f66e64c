"""Statistics, lattice snap and shift lists of a build at the edges of their kernels: one block or
several, index ranges of one tile, of as many as one launch compacts and of one more, values next
to the half-way points of the lattice, against the oracle's snap and plain numpy."""

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

TILE = 4096


@pytest.mark.parametrize("n,span", [(8, 1), (64, TILE), (64, TILE + 1), (128, 48 * TILE),
                                    (128, 48 * TILE + 1), (256, 300_000)])
def test_per_point_shift_lists(n, span):
    """Every point's shift is the oracle's snap of its value (whole numbers: no tolerance), the list
    is their sorted set, for index ranges of `span` with values up to 1e-9 from the half-way points
    (where the answer turns on the last bits of the plain evaluation)."""
    import torch
    from paper_1607_02560_gb300 import Context
    rng = np.random.default_rng(n + span)
    N = n * n
    m = rng.integers(0, span, size=N)
    m[0], m[-1] = 0, span - 1
    near = 10.0 ** rng.uniform(-9, 0, size=N) * 0.5
    frac = np.where(rng.random(N) < 0.5, 0.5 - near, rng.uniform(-0.49, 0.49, size=N))
    frac *= np.sign(rng.uniform(-1, 1, size=N))
    frac[m == 0] = np.abs(frac[m == 0])
    frac[m == span - 1] = -np.abs(frac[m == span - 1])
    if span == 1:
        frac[:] = rng.uniform(-0.4, 0.4, size=N)
    v = ((4.0 * (m + frac) + 2.0) * O.PI2).reshape(n, n)
    want = np.asarray(O.snap_index(v.reshape(-1)), dtype=np.int64)
    ctx = Context(2, n, stream=torch.cuda.Stream())
    ctx.set_potential(v)
    ctx.build_stencils(policy="local")
    t = ctx.get_shift_table()
    shifts = np.sort(np.unique(want))
    assert np.array_equal(t["s"], np.array([O.shift_value(int(k)) for k in shifts]))
    assert np.array_equal(shifts[t["s_idx"]], want)


@pytest.mark.parametrize("n", [8, 64, 512])
def test_statistics_refuse_non_finite_values(n):
    """One bad value anywhere is found, by one block (n = 8) or several (n = 64, 512)."""
    import torch
    from paper_1607_02560_gb300 import Context
    from paper_1607_02560_gb300.lsp import LspError
    rng = np.random.default_rng(n)
    ctx = Context(2, n, stream=torch.cuda.Stream())
    for bad, at in ((np.nan, 0), (np.inf, n * n - 1), (-np.inf, n * n // 2)):
        v = rng.standard_normal(n * n)
        v[at] = bad
        with pytest.raises(LspError):
            ctx.set_potential(v.reshape(n, n))
    ctx.set_potential(rng.standard_normal((n, n)))


@pytest.mark.parametrize("n,ns,spread", [(8, 1, 0), (64, 2, 1), (64, 3, 5000), (128, 64, 1000)])
def test_nearest_of_a_shift_list(n, ns, spread):
    """Every point takes the listed shift nearest to its value, ties to the smaller: the oracle's
    assignment, with values on the shifts, half-way between neighbours and next to both."""
    import torch
    from paper_1607_02560_gb300 import Context
    rng = np.random.default_rng(n + ns)
    N = n * n
    m = np.sort(rng.choice(np.arange(0, max(spread, ns) + 1), size=ns, replace=False)) + 3
    s = np.asarray(O.shift_value(m))
    k = rng.integers(0, ns, size=N)
    near = 10.0 ** rng.uniform(-16, 0, size=N) * np.sign(rng.uniform(-1, 1, size=N))
    mid = 0.5 * (s[k] + s[np.minimum(k + 1, ns - 1)])
    v = np.where(rng.random(N) < 0.5, s[k], mid) * np.where(rng.random(N) < 0.2, 1.0, 1.0 + near)
    v = np.where(rng.random(N) < 0.3, rng.uniform(s[0] - 100, s[-1] + 100, size=N), v)
    want = np.asarray(O.assign_shifts(v, m)).reshape(-1)
    ctx = Context(2, n, stream=torch.cuda.Stream())
    ctx.set_potential(v.reshape(n, n))
    ctx.build_stencils(policy="list", shifts=s)
    t = ctx.get_shift_table()
    assert np.array_equal(t["s"], s)
    assert np.array_equal(t["s_idx"], want)
