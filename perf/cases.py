"""The work that users of the library have it do, as timed cases.

Every case goes through the public Python binding the way a program uses it: a context (and, for
the solves, a factorisation) is made once for a grid; each pass brings a potential or a
right-hand side that lives on the GPU and takes the results as GPU tensors. Potentials are seeded
fields of the shapes the library is built for: Helmholtz velocity bumps in 1D and 2D, Schroedinger
wells in 3D.

Kinds:
  build     set_potential + build_stencils + the Q, C and P rows
  operator  y = (L + diag v) u
  factor    nested-dissection factorisation of P and one solve with it
  gmres     the preconditioned GMRES solve of (L + diag v) u = f
  train     one training step of the learned stencils' network
"""

import functools
import itertools
import math

import numpy as np
import torch

import paper_1607_02560_gb300 as lsp

PI2 = math.pi * math.pi
F64 = torch.float64


def listed():
    return [
        # the smallest whole build: the 32 x 32 demonstration problem, where launches count
        dict(name="build_fp64_2d_n32", kind="build", d=2, n=32, mode="fp64", policy="local",
             bumps=1, ppw=4.0),
        # the headline workload: every point its own shift, a million points, FP64
        dict(name="build_fp64_2d_n1024", kind="build", d=2, n=1024, mode="fp64", policy="local",
             bumps=64, ppw=4.0),
        # the same build in the mixed precision mode
        dict(name="build_mixed_2d_n1024", kind="build", d=2, n=1024, mode="mixed",
             policy="local", bumps=64, ppw=4.0),
        # an ordinary 2D build in double words
        dict(name="build_dword_2d_n256", kind="build", d=2, n=256, mode="dword", policy="local",
             bumps=16, ppw=4.0),
        # rows from the learned network, a million points
        dict(name="build_learned_2d_n1024", kind="build", d=2, n=1024, mode="learned",
             policy="local", bumps=64, ppw=4.0),
        # the 3D workload: 27-point rows, few shifts
        dict(name="build_fp64_3d_n64", kind="build", d=3, n=64, mode="fp64", policy="local",
             bumps=8, ppw=4.0),
        # wide and narrow rows by distance to the separators, an odd number of shifts
        dict(name="build_multit_2d_n128", kind="build", d=2, n=128, mode="fp64", policy="paper",
             nshifts=13, t=2, leaf=8, bumps=16, ppw=6.0),
        # one application of the pseudospectral operator (a matrix-free solver's inner call)
        dict(name="operator_2d_n1024", kind="operator", d=2, n=1024, bumps=64, ppw=4.0),
        # factorisation and a refined solve: many small fronts
        dict(name="factor_2d_n512", kind="factor", d=2, n=512, policy="paper", nshifts=32,
             leaf=8, refine=1, bumps=1, ppw=4.0),
        # factorisation and a refined solve: few large fronts
        dict(name="factor_3d_n32", kind="factor", d=3, n=32, policy="paper", nshifts=8, leaf=8,
             refine=1, bumps=8, ppw=4.0),
        # the whole preconditioned solve at the largest 2D grid, factor in hand
        dict(name="gmres_2d_n1024", kind="gmres", d=2, n=1024, policy="paper", nshifts=64,
             leaf=8, refine=1, bumps=16, ppw=4.0),
        # one step of the training loop that makes the learned stencils
        dict(name="train_2d_b4096", kind="train", d=2, n=256, batch=4096, bumps=16, ppw=4.0),
    ]


def draw(rng):
    kind = rng.choice(["build", "build", "build", "learned", "multit", "operator", "factor",
                       "gmres", "train"])
    bumps = rng.randint(1, 64)
    ppw = round(rng.uniform(4.0, 9.0), 2)
    if kind == "build":
        d = rng.choice([1, 2, 2, 2, 3, 3])
        n = 2 ** (rng.randint(5, 12) if d == 1 else rng.randint(4, 10) if d == 2
                  else rng.randint(3, 6))
        c = dict(kind="build", d=d, n=n, mode=rng.choice(["fp64", "fp64", "mixed", "dword"]),
                 policy=rng.choice(["local", "local", "paper"]), bumps=bumps, ppw=ppw)
        if c["policy"] == "paper":
            c["nshifts"] = rng.randint(3, 101)
        return c
    if kind == "learned":
        d = rng.choice([2, 3])
        return dict(kind="build", d=d, n=2 ** (rng.randint(5, 10) if d == 2 else rng.randint(3, 6)),
                    mode="learned", policy="local", bumps=bumps, ppw=ppw)
    if kind == "multit":
        return dict(kind="build", d=2, n=2 ** rng.randint(5, 7), mode="fp64", policy="paper",
                    nshifts=rng.randint(3, 41), t=2, leaf=rng.choice([4, 8, 16]), bumps=bumps,
                    ppw=round(rng.uniform(5.0, 9.0), 2))
    if kind == "operator":
        d = rng.choice([1, 2, 3])
        n = 2 ** (rng.randint(6, 12) if d == 1 else rng.randint(4, 10) if d == 2
                  else rng.randint(3, 6))
        return dict(kind="operator", d=d, n=n, bumps=bumps, ppw=ppw)
    if kind == "factor":
        d = rng.choice([2, 2, 3])
        n = 2 ** (rng.randint(5, 9) if d == 2 else rng.randint(3, 5))
        leaf = 4 if n == 8 else rng.choice([4, 8, 8, 16] if d == 2 else [4, 8])
        return dict(kind="factor", d=d, n=n, policy=rng.choice(["paper", "local"]),
                    nshifts=rng.randint(5, 41), leaf=leaf, refine=1, bumps=bumps, ppw=ppw)
    if kind == "gmres":
        d = rng.choice([2, 2, 3])
        n = 2 ** (rng.randint(5, 9) if d == 2 else rng.randint(4, 5))
        return dict(kind="gmres", d=d, n=n, policy="paper", leaf=8, refine=1,
                    nshifts=(max(4, n // 16) if d == 2 else n // 4) + rng.randint(0, 5),
                    bumps=rng.randint(4, 24), ppw=ppw)
    d = rng.choice([2, 3])
    return dict(kind="train", d=d, n=64 if d == 2 else 16,
                batch=128 * int(round(2 ** rng.uniform(0.0, 5.0))), bumps=bumps, ppw=ppw)


# ---- inputs -------------------------------------------------------------------------------------

def _axes(n, d):
    x = torch.arange(n, dtype=F64, device="cuda") / n
    return [x.reshape([n if a == b else 1 for b in range(d)]) for a in range(d)]


def _field(n, d, amps, centres, widths):
    """Sum of periodic Gaussians amp exp(-|x - x_j|^2 / (2 w^2)) on the n^d grid."""
    ax = _axes(n, d)
    f = torch.zeros([n] * d, dtype=F64, device="cuda")
    for a, xc, w in zip(amps, centres, widths):
        prod = None
        for x, c in zip(ax, xc):
            delta = torch.remainder(x - c + 0.5, 1.0) - 0.5
            e = torch.exp(-delta * delta / (2.0 * w * w))
            prod = e if prod is None else prod * e
        f += a * prod
    return f


def _potential(case, seed):
    """v on the grid: -(omega / c)^2 in 1D and 2D, wells of depth max|v| h^2 = 9.6 / ppw^2 in 3D."""
    rng = np.random.default_rng([seed, 1])
    d, n, nb = case["d"], case["n"], case["bumps"]
    if d == 3:
        base = -_field(n, d, rng.uniform(0.5, 1.5, nb), rng.uniform(0.0, 1.0, (nb, d)),
                       [0.05] * nb) - 0.3
        target = 9.6 / case["ppw"] ** 2
        return (base * (target * n * n / base.abs().max())).contiguous()
    if nb == 1:  # a single centred lens of slower or faster medium
        bump = _field(n, d, [rng.uniform(0.1, 0.3)], [[0.5] * d], [rng.uniform(0.08, 0.12)])
    else:
        bump = _field(n, d, rng.uniform(-0.3, 0.3, nb), rng.uniform(0.0, 1.0, (nb, d)),
                      rng.uniform(0.02, 0.08, nb))
    low = float(bump.min())
    if low < -0.6:  # the velocity stays positive
        bump *= -0.6 / low
    omega = 2.0 * math.pi * n / case["ppw"]
    return (-(omega / (1.0 + bump)) ** 2).contiguous()


def _smooth(case, seed):
    """A band-limited wave packet: a grid function with structure at several scales."""
    rng = np.random.default_rng([seed, 2])
    d, n = case["d"], case["n"]
    ax = _axes(n, d)
    u = torch.zeros([n] * d, dtype=F64, device="cuda")
    for _ in range(6):
        k = rng.integers(-(n // 8), n // 8 + 1, d)
        phase = sum(2.0 * math.pi * int(ki) * x for ki, x in zip(k, ax)) + rng.uniform(0, 6.28)
        u = u + rng.uniform(0.5, 1.5) * torch.cos(phase)
    return u.reshape(-1).contiguous()


def _apply(v, u):
    """(L + diag v) u by a full complex transform."""
    n, d = v.shape[0], v.dim()
    k = torch.fft.fftfreq(n, d=1.0 / n, dtype=F64, device=v.device)
    k2 = sum((k * k).reshape([n if a == b else 1 for b in range(d)]) for a in range(d))
    x = u.reshape(v.shape)
    return (torch.fft.ifftn(4.0 * PI2 * k2 * torch.fft.fftn(x)).real + v * x).reshape(-1)


def _shifted(x, offs):
    """x[(j + o) mod n] for every offset o, one column per offset."""
    dims = list(range(x.dim()))
    return torch.stack([torch.roll(x, [-int(c) for c in o], dims).reshape(-1) for o in offs], 1)


def _offsets(d, t):
    return list(itertools.product(range(-t, t + 1), repeat=d))


def _snap(x):
    """Index m of the lattice shift (4 m + 2) pi^2 nearest to x, halves away from zero."""
    y = (x / PI2 - 2.0) * 0.25
    r = torch.trunc(y)
    return (r + torch.sign(y) * ((y - r).abs() >= 0.5)).to(torch.int64)


def _lattice(m):
    return (4 * m + 2).to(F64) * PI2


@functools.lru_cache(maxsize=None)
def _stream():
    return torch.cuda.Stream()


def _net(d):
    """Sizes of the network: inputs, padded inputs, outputs, padded outputs."""
    return (26, 32, 18, 32) if d == 2 else (126, 128, 54, 64)


def _params(case, seed, v):
    """A network's flat parameter vector: the weights of a freshly started fit, normalised for the
    stencils of v (mean stencil plus a small learned part)."""
    rng = np.random.default_rng([seed, 3])
    d, n = case["d"], case["n"]
    nf, k0, out, outp = _net(d)
    mu, h2 = out // 2, 1.0 / (n * n)
    parts = []
    for rows, cols, live_r, live_c, scale in ((256, k0, 256, nf, 1.0), (256, 256, 256, 256, 1.0),
                                              (256, 256, 256, 256, 1.0),
                                              (outp, 256, out, 256, 0.5)):
        w = np.zeros((rows, cols), np.float32)
        a = scale * math.sqrt(6.0 / live_c)
        w[:live_r, :live_c] = rng.uniform(-a, a, (live_r, live_c))
        b = np.zeros(rows, np.float32)
        b[:live_r] = rng.uniform(-0.05, 0.05, live_r)
        parts += [w.ravel(), b]
    x = v * h2
    lo, hi = float(x.min()), float(x.max())
    order = np.abs(np.array(_offsets(d, 1))).sum(1)
    mean = np.concatenate([np.array([0.88, -0.19, 0.04, -0.01])[order],
                           np.array([0.10, 0.02, 0.004, 0.001])[order] * h2]).astype(np.float32)
    sig = np.concatenate([np.full(mu, 0.02), np.full(mu, 0.002 * h2)]).astype(np.float32)
    pad = outp - out
    parts += [np.array([0.5 * (lo + hi), 0.3 * (hi - lo) + 1e-3], np.float32),
              mean, np.zeros(pad, np.float32), sig, np.ones(pad, np.float32),
              np.array([lo - 0.01 * (hi - lo) - 1e-6, hi + 0.01 * (hi - lo) + 1e-6], np.float32)]
    return np.concatenate(parts).astype(np.float32)


def _pairs(case, seed, v):
    """Raw training pairs at random points: the 5^d patch of h^2 v and h^2 s_j, and stencils that
    follow it smoothly."""
    d, n, batch = case["d"], case["n"], case["batch"]
    nf, _, out, _ = _net(d)
    g = torch.Generator(device="cuda").manual_seed(1000 + seed)
    j = torch.randint(0, n ** d, (batch,), generator=g, device="cuda")
    h2 = 1.0 / (n * n)
    patch = _shifted(v, _offsets(d, 2))[j]
    x = torch.cat([patch, _lattice(_snap(v.reshape(-1)[j]))[:, None]], 1) * h2
    mix = torch.randn(nf, out, generator=g, dtype=F64, device="cuda") / math.sqrt(nf)
    z = torch.tanh((x - x.mean()) / (x.std() + 1e-12) @ mix)
    flat = torch.from_numpy(_params(case, seed, v)).cuda().to(F64)
    _, _, _, outp = _net(d)
    stats = flat[-(2 + 2 * outp) - 2:]
    mean, sig = stats[2:2 + out], stats[2 + outp:2 + outp + out]
    return x.float().contiguous(), (mean + sig * z).float().contiguous()


# ---- prepare and run ----------------------------------------------------------------------------

def _build_args(case):
    a = dict(policy=case["policy"], mode=case.get("mode", "fp64"), use_graph=True,
             t=case.get("t", 1), nd_leaf=case["leaf"] if case.get("t", 1) == 2 else 0)
    if case["policy"] == "paper":
        a["nshifts"] = case["nshifts"]
    return a


def prepare(case, seed):
    d, n = case["d"], case["n"]
    v = _potential(case, seed)
    st = {"case": case, "v": v}
    if case["kind"] == "train":
        st["X"], st["T"] = _pairs(case, seed, v)
        torch.cuda.synchronize()
        st["mlp"] = lsp.Mlp(d, seed=0, stream=_stream())
        st["mlp"].set_params(_params(case, seed, v))
        st["grads"] = np.empty(st["mlp"].nweights, np.float32)
        return st
    torch.cuda.synchronize()
    ctx = st["ctx"] = lsp.Context(d, n, stream=_stream())
    if case["kind"] == "build":
        mu = (2 * case.get("t", 1) + 1) ** d
        st["rows"] = {w: torch.empty((n ** d, mu), dtype=F64, device="cuda") for w in "QCP"}
        st["args"] = _build_args(case)
        if case["mode"] == "learned":
            st["mlp"] = lsp.Mlp(d, seed=0, stream=_stream())
            st["mlp"].set_params(_params(case, seed, v))
            ctx.set_mlp(st["mlp"])
        torch.cuda.synchronize()
        return st
    ctx.set_potential(v)
    st["out"] = torch.empty(n ** d, dtype=F64, device="cuda")
    if case["kind"] == "operator":
        st["u"] = _smooth(case, seed)
        torch.cuda.synchronize()
        return st
    a = _build_args(case)
    ctx.build_stencils(**a)
    ctx.nd_factor(leaf=case["leaf"], refine_steps=case["refine"])
    if case["kind"] == "factor":
        rows = torch.empty((n ** d, ctx.mu), dtype=F64, device="cuda")
        torch.cuda.synchronize()
        ctx.get_rows("P", rows)
        ctx.synchronize()
        near = _shifted(_smooth(case, seed).reshape([n] * d), _offsets(d, 1))
        st["y"] = (rows * near).sum(1).contiguous()
    else:
        st["f"] = _apply(v, _smooth(case, seed)).contiguous()
    torch.cuda.synchronize()
    return st


def run(state):
    kind = state["case"]["kind"]
    if kind == "build":
        ctx = state["ctx"]
        ctx.set_potential(state["v"])
        ctx.build_stencils(**state["args"])
        return {w: ctx.get_rows(w, state["rows"][w]) for w in "QCP"}
    if kind == "operator":
        state["ctx"].apply_operator(state["u"], state["out"])
        return {"y": state["out"]}
    if kind == "factor":
        case, ctx = state["case"], state["ctx"]
        ctx.nd_factor(leaf=case["leaf"], refine_steps=case["refine"])
        ctx.nd_solve(state["y"], state["out"])
        return {"x": state["out"]}
    if kind == "gmres":
        u, res = state["ctx"].gmres(state["f"], state["out"], max_cycles=2)
        return {"u": u, "iterations": res["iterations"]}
    case, mlp = state["case"], state["mlp"]
    loss = mlp.train_step(state["X"], state["T"], case["batch"], 1e-5, apply=True,
                          grads=state["grads"])
    return {"loss": np.float32(loss), "grads": state["grads"]}


# ---- work ---------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _plan(d, n, leaf):
    return lsp.lsp.nd_plan_info(n, leaf=leaf, d=d)


def work(case):
    """Bytes of the inputs and outputs, and the operations of the smallest known method."""
    d, n = case["d"], case["n"]
    N, mu = n ** d, (2 * case.get("t", 1) + 1) ** d
    nf, _, out, _ = _net(max(d, 2))
    net = 2.0 * (nf * 256 + 2 * 256 * 256 + 256 * out)
    kind = case["kind"]
    if kind == "build":
        flops = N * net if case["mode"] == "learned" else 2.0 * mu * N
        return {"bytes": 8.0 * N * (1 + 3 * mu), "flops": flops}
    if kind == "operator":
        return {"bytes": 24.0 * N, "flops": 5.0 * N * math.log2(N) + 3.0 * N}
    if kind == "factor":
        p = _plan(d, n, case["leaf"])
        return {"bytes": 8.0 * N * (mu + 2) + p["solve_bytes"],
                "flops": p["flops_lu"] + p["solve_bytes"] / 4.0}
    if kind == "gmres":  # at least four applications of P^-1, C and the operator
        p = _plan(d, n, case["leaf"])
        return {"bytes": 4.0 * (p["solve_bytes"] + 8.0 * N * (mu + 8)),
                "flops": 4.0 * (p["solve_bytes"] / 4.0 + N * (2.0 * mu + 5.0 * math.log2(N)))}
    B = case["batch"]
    weights = nf * 256 + 2 * 256 * 256 + 256 * out
    return {"bytes": 4.0 * (B * (nf + out) + 6.0 * weights), "flops": 3.0 * B * net}


# ---- the same outputs in 64 bits ------------------------------------------------------------------

def _green(n, d, amax, ms):
    """g_s and g_s * g_s at offsets 0..amax along every axis, for the lattice shifts of index ms:
    [len(ms), 2, amax + 1, ...], the inverse transform summed one axis at a time."""
    A = amax + 1
    p = torch.arange(n // 2 + 1, dtype=torch.int64, device="cuda")
    wgt = torch.full((n // 2 + 1,), 2.0, dtype=F64, device="cuda")
    wgt[0] = wgt[-1] = 1.0
    X = torch.stack([wgt * torch.cos(2.0 * math.pi * ((a * p) % n).to(F64) / n)
                     for a in range(A)], 1)
    p2 = p * p
    lo, hi = int(ms.min()), int(ms.max())
    top = (n // 2) ** 2
    w = 1.0 / _lattice(torch.arange(lo, hi + d * top + 1, device="cuda"))
    table = torch.stack([w, w * w])[None]  # [classes, 2, range]
    for k in range(1, d + 1):
        ls = ms if k == d else torch.arange(lo, hi + (d - k) * top + 1, device="cuda")
        step = max(1, int(6e7) // (table.shape[0] * 2 * len(p2)))
        parts = [torch.einsum("cflp,pa->acfl", table[:, :, l[:, None] - lo + p2[None, :]], X)
                 for l in ls.split(step)]
        table = torch.cat(parts, 3).reshape(A * table.shape[0], 2, len(ls))
    return (table / float(n) ** d).permute(2, 1, 0).reshape([len(ms), 2] + [A] * d)


def _stencils(n, d, t, ms):
    """alpha and c of every lattice shift in ms, [len(ms), (2t+1)^d] each."""
    g = _green(n, d, 2 * t, ms).cpu().numpy()
    offs = np.array(_offsets(d, t))
    diff = np.abs(offs[:, None, :] - offs[None, :, :])
    pick = tuple(diff[:, :, a] for a in range(d))
    alpha, c = [], []
    for chunk in np.array_split(g, max(1, len(g) // 4096)):
        G, A1 = chunk[(slice(None), 0) + pick], chunk[(slice(None), 1) + pick]
        _, vec = np.linalg.eigh(A1 - G @ G)
        a = vec[:, :, 0]
        a = a * np.where(a[:, [len(offs) // 2]] < 0, -1.0, 1.0)
        alpha.append(a)
        c.append(np.einsum("sab,sb->sa", G, a))
    return (torch.from_numpy(np.concatenate(x)).cuda() for x in (alpha, c))


def _shift_list(case, v):
    """Lattice indices of the shifts in use, and each point's position among them."""
    m = _snap(v.reshape(-1))
    if case["policy"] == "local":
        return torch.unique(m, return_inverse=True)
    lo, hi, K = float(v.min()), float(v.max()), case["nshifts"]
    xs = [lo + i * ((hi - lo) / (K - 1)) for i in range(K - 1)] + [hi]
    ms = torch.unique(_snap(torch.tensor(xs, dtype=F64, device="cuda")))
    s, x = _lattice(ms), v.reshape(-1)
    right = torch.searchsorted(s, x).clamp(max=len(s) - 1)
    left = (right - 1).clamp(min=0)
    return ms, torch.where((s[left] - x).abs() <= (s[right] - x).abs(), left, right)


def _exact_rows(case, v):
    d, n, t = case["d"], case["n"], case.get("t", 1)
    ms, idx = _shift_list(case, v)
    s = _lattice(ms)[idx][:, None]
    Q, C = (x[idx] for x in _stencils(n, d, t, ms))
    if t == 2:  # points near a separator keep the 3^d stencil in the inner columns
        leaf, offs = case["leaf"], np.array(_offsets(d, 2))
        inner = torch.from_numpy(np.flatnonzero((np.abs(offs) <= 1).all(1))).cuda()
        r = torch.arange(n, device="cuda") % leaf
        f = torch.where(r == 0, torch.full_like(r, leaf), torch.minimum(r, leaf - r))
        near = torch.stack([f.reshape([n if a == b else 1 for b in range(d)]).expand([n] * d)
                            for a in range(d)]).amin(0).reshape(-1) < 2
        for full, small in zip((Q, C), _stencils(n, d, 1, ms)):
            part = torch.zeros((int(near.sum()), full.shape[1]), dtype=F64, device="cuda")
            part[:, inner] = small[idx[near]]
            full[near] = part
    return {"Q": Q, "C": C, "P": Q + C * (_shifted(v, _offsets(d, t)) - s)}


def _layers(case, seed, v):
    """Weights (rounded to the bf16 that the network holds), biases and normalisation."""
    flat = torch.from_numpy(_params(case, seed, v)).cuda()
    nf, k0, out, outp = _net(case["d"])
    at, layers = 0, []
    for rows, cols in ((256, k0), (256, 256), (256, 256), (outp, 256)):
        w = flat[at:at + rows * cols].reshape(rows, cols).bfloat16().to(F64)
        b = flat[at + rows * cols:at + rows * cols + rows].to(F64)
        at += rows * cols + rows
        layers += [w, b]
    tail = flat[at:].to(F64)
    return layers, tail[0], tail[1], tail[2:2 + out], tail[2 + outp:2 + outp + out]


def _forward(layers, x):
    for k in range(0, 8, 2):
        x = x @ layers[k].T + layers[k + 1]
        if k < 6:
            x = torch.relu(x)
    return x


def _features(case, x, mu, sig):
    nf, k0, _, _ = _net(case["d"])
    x = ((x - mu) / sig).bfloat16().to(F64)
    return torch.nn.functional.pad(x, (0, k0 - nf))


def _exact_learned(case, seed, v):
    d, n = case["d"], case["n"]
    h2, out = 1.0 / (n * n), _net(d)[2]
    layers, mu, sig, my, sy = _layers(case, seed, v)
    s = _lattice(_snap(v.reshape(-1)))[:, None]
    x = torch.cat([_shifted(v, _offsets(d, 2)), s], 1) * h2
    y = torch.cat([_forward(layers, _features(case, c, mu, sig))[:, :out] * sy + my
                   for c in x.split(1 << 17)])
    norm = y[:, :out // 2].norm(dim=1, keepdim=True)
    Q, C = y[:, :out // 2] / norm, y[:, out // 2:] / norm
    return {"Q": Q, "C": C, "P": Q + C * (_shifted(v, _offsets(d, 1)) - s)}


def _exact_train(case, seed, v):
    X, T = _pairs(case, seed, v)
    out = _net(case["d"])[2]
    layers, mu, sig, my, sy = _layers(case, seed, v)
    for w in layers:
        w.requires_grad_(True)
    y = _forward(layers, _features(case, X.to(F64), mu, sig))[:, :out]
    loss = ((y - (T.to(F64) - my) / sy) ** 2).mean()
    loss.backward()
    return {"loss": float(loss), "grads": torch.cat([w.grad.reshape(-1) for w in layers])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "factor":  # y was formed as P x
        return {"x": _smooth(case, seed)}
    if kind == "gmres":   # f was formed as (L + diag v) u
        return {"u": _smooth(case, seed), "iterations": None}
    v = _potential(case, seed)
    if kind == "operator":
        return {"y": _apply(v, _smooth(case, seed))}
    if kind == "train":
        return _exact_train(case, seed, v)
    return _exact_learned(case, seed, v) if case["mode"] == "learned" else _exact_rows(case, v)
