"""Performance cases: the sweeps a user of the library runs, through its
public Python entry points.

A case is a dict of plain values.  "kind" is one of
  const    Plan(shape, radius, weights, boundary).run(grid, steps)
  batch    Batch(grids, alphas, steps).run(): many uneven 2D heat grids
  diffuse  autograd.diffuse and its backward pass (variable coefficients)
Every pass starts from the same initial field (a copy of it is advanced), so
a pass does the same work however often it is repeated.
"""
import math
import random

import numpy as np
import torch

import paper_2303_08365_gb300 as st
from paper_2303_08365_gb300 import autograd as st_autograd


def const(name, shape, stencil, weights, periodic, steps, field, alpha=0.1):
    """stencil: star or box and its radius, as in "star1"; shape: slowest axis first."""
    return {"name": name, "kind": "const", "ndim": len(shape), "n0": shape[0],
            "n1": shape[1] if len(shape) > 1 else 1, "n2": shape[2] if len(shape) > 2 else 1,
            "stencil": stencil, "weights": weights, "alpha": alpha, "periodic": periodic, "steps": steps,
            "field": field}


def listed():
    return [
        # the smallest simulation: a 256 x 256 heat plate advanced 100 steps, where launches and latency count
        const("heat2d 256", (256, 256), "star1", "heat", False, 100, "uniform"),
        # an ordinary plate, between the small grids and the ones that fill the chip
        const("heat2d 1000", (1000, 1000), "star1", "heat", False, 100, "uniform"),
        # the copper plate of the thermal study, a hot spot on a cold plate, over an odd number of steps
        const("plate2d 9600", (9600, 9600), "star1", "heat", False, 21, "spot", 0.23),
        # repeated 3 x 3 smoothing of a large periodic image
        const("box2d equal 16384", (16384, 16384), "box1", "equal", True, 10, "uniform"),
        # a radius-2 kernel with general weights (Box-2D25P)
        const("box2d25 8192", (8192, 8192), "box2", "random", True, 4, "normal"),
        # the headline simulation: 3D heat, periodic, 512 cubed
        const("heat3d 512", (512, 512, 512), "star1", "heat", True, 20, "uniform"),
        # a small 3D box, many short steps
        const("heat3d 64", (64, 64, 64), "star1", "heat", True, 100, "uniform"),
        # 27 general weights on zero-mean data
        const("box3d27 384", (384, 384, 384), "box1", "random", False, 4, "normal"),
        # a 3D grid whose sizes are not multiples of anything, general star weights
        const("star3d odd", (199, 251, 301), "star1", "random", False, 21, "normal"),
        # the long 1D rod of Heat-1D
        const("heat1d 1e7", (10_000_000,), "star1", "heat", False, 40, "uniform"),
        # many independent plates of uneven sizes and step counts in one call
        {"name": "batch 48 plates", "kind": "batch", "grids": 48, "lo": 128, "hi": 4096, "t_lo": 5, "t_hi": 50,
         "layout": 2307, "periodic": False},
        # fitting a conductivity field: forward sweep and gradients for u0 and kappa
        {"name": "diffuse 3d 192", "kind": "diffuse", "ndim": 3, "n0": 192, "n1": 192, "n2": 192, "periodic": True,
         "steps": 60, "ckpt": 0},
    ]


def log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same families: sizes log-uniform, odd ones among
    them, steps chosen so that it costs no more than the largest listed case."""
    kind = rng.choice(["const2"] * 4 + ["const3"] * 4 + ["const1", "batch", "diffuse"])
    periodic = rng.random() < 0.5
    if kind == "batch":
        lo = log_int(rng, 32, 256)
        return {"kind": "batch", "grids": rng.randint(4, 60), "lo": lo, "hi": log_int(rng, lo, 2048),
                "t_lo": rng.randint(1, 20), "t_hi": rng.randint(20, 60), "layout": rng.randint(1, 10**6),
                "periodic": periodic}
    if kind == "diffuse":
        if rng.random() < 0.5:
            a, b = log_int(rng, 64, 1500), log_int(rng, 64, 1500)
            return {"kind": "diffuse", "ndim": 2, "n0": a, "n1": b, "n2": 1, "periodic": periodic,
                    "steps": rng.randint(4, 60), "ckpt": rng.choice([0, 1, 8])}
        n = [log_int(rng, 24, 192) for _ in range(3)]
        return {"kind": "diffuse", "ndim": 3, "n0": n[0], "n1": n[1], "n2": n[2], "periodic": periodic,
                "steps": rng.randint(4, 50), "ckpt": rng.choice([0, 1, 8])}
    weights = rng.choice(["heat", "random", "random", "equal"])
    radius = 1 if weights == "heat" else rng.choice([1, 1, 2])
    if kind == "const1":
        shape, stencil = (log_int(rng, 1000, 10_000_000),), "star%d" % radius
        weights = "random" if weights == "equal" else weights
    elif kind == "const2":
        shape = (log_int(rng, 64, 10000), log_int(rng, 64, 10000))
        stencil = ("star" if weights == "heat" else rng.choice(["star", "box"])) + str(radius)
    else:
        shape = tuple(log_int(rng, 24, 400) for _ in range(3))
        stencil = ("star" if weights == "heat" else rng.choice(["star", "box"])) + str(radius)
    if weights == "equal":
        stencil = "box%d" % radius
    if rng.random() < 0.4:  # sizes that the tiles like as well as ragged ones
        shape = tuple(max(64, n // 64 * 64) for n in shape)
    cells, taps = int(np.prod(shape)), n_taps(stencil, len(shape))
    most = int(2e10 / (cells * taps)) // (4 if taps > 30 else 1)
    return const("", shape, stencil, weights, periodic, max(1, min(rng.randint(1, 100), most)),
                 rng.choice(["uniform", "normal", "spot"]), rng.uniform(0.05, 0.16)) | {"name": "drawn"}


# ------------------------------------------------------------------ inputs


def shape_of(case):
    return tuple(case["n%d" % d] for d in range(case["ndim"]))


def n_taps(stencil, ndim):
    r = int(stencil[-1])
    return 2 * ndim * r + 1 if stencil.startswith("star") else (2 * r + 1) ** ndim


def weights_of(case):
    """The dense weight array of a const case (the same for every seed)."""
    nd, r = case["ndim"], int(case["stencil"][-1])
    side = 2 * r + 1
    off = np.stack(np.meshgrid(*[np.arange(-r, r + 1)] * nd, indexing="ij"))
    star = (off != 0).sum(axis=0) <= 1
    w = np.zeros((side,) * nd)
    if case["weights"] == "heat":
        a = case["alpha"] if nd < 3 else min(case["alpha"], 0.16)
        w[star] = a
        w[(r,) * nd] = 1.0 - 2 * nd * a
    elif case["weights"] == "equal":
        w[...] = 1.0 / side ** nd
    else:
        w = np.random.default_rng(1000 * nd + 10 * r + case["stencil"].startswith("star")).random((side,) * nd)
        if case["stencil"].startswith("star"):
            w[~star] = 0.0
        w /= w.sum()
    return w


def field(kind, shape, gen):
    if kind == "uniform":
        return torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda")
    if kind == "normal":
        return torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda")
    # a Gaussian hot spot (100 degrees) somewhere near the middle of a cold domain
    u = torch.full((), 100.0, dtype=torch.float64, device="cuda")
    at = torch.rand(len(shape), generator=gen, dtype=torch.float64, device="cuda")
    for d, n in enumerate(shape):
        x = torch.arange(n, dtype=torch.float64, device="cuda") - n * (0.4 + 0.2 * at[d])
        u = u[..., None] * torch.exp(-0.5 * (x / (0.143 * n)) ** 2)
    return u.contiguous()


def generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def layout(case):
    """Sizes, alphas and step counts of a batch (fixed by the case, not by the seed)."""
    r = random.Random(case["layout"])
    return [(log_int(r, case["lo"], case["hi"]), log_int(r, case["lo"], case["hi"]), r.uniform(0.05, 0.24),
             r.randint(case["t_lo"], case["t_hi"])) for _ in range(case["grids"])]


def diffuse_inputs(case, seed):
    gen, shape = generator(seed), shape_of(case)
    u0 = torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda")
    kappa = torch.exp(0.5 * torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda"))
    grad = torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda")
    return u0, kappa, grad, 0.1 / float(kappa.max())


def prepare(case, seed):
    periodic = st.PERIODIC if case["periodic"] else st.DIRICHLET_ZERO
    if case["kind"] == "batch":
        gen, items = generator(seed), layout(case)
        u0 = [torch.rand(ny, nx, generator=gen, dtype=torch.float64, device="cuda") for ny, nx, _, _ in items]
        grids = [torch.empty_like(u) for u in u0]
        batch = st.Batch(grids, [a for _, _, a, _ in items], [t for _, _, _, t in items], periodic)
        return {"kind": "batch", "u0": u0, "grids": grids, "batch": batch}
    if case["kind"] == "diffuse":
        u0, kappa, grad, dt = diffuse_inputs(case, seed)
        return {"kind": "diffuse", "u0": u0.requires_grad_(), "kappa": kappa.requires_grad_(), "grad": grad, "dt": dt,
                "plan": st.Plan.varcoef(shape_of(case), periodic), "steps": case["steps"], "ckpt": case["ckpt"]}
    shape = shape_of(case)
    return {"kind": "const", "u0": field(case["field"], shape, generator(seed)), "steps": case["steps"],
            "plan": st.Plan(shape, int(case["stencil"][-1]), weights_of(case), periodic)}


def run(state):
    if state["kind"] == "batch":
        torch._foreach_copy_(state["grids"], state["u0"])
        state["batch"].run()
        return state["grids"]
    if state["kind"] == "diffuse":
        out = st_autograd.diffuse(state["u0"], state["kappa"], state["plan"], state["dt"], state["steps"],
                                  state["ckpt"])
        return [out.detach(), *torch.autograd.grad(out, (state["u0"], state["kappa"]), state["grad"])]
    return state["plan"].run(state["u0"].clone(), state["steps"])


def work(case):
    """Each field read once and written once; 2K-1 flops for a K-tap update."""
    if case["kind"] == "batch":
        items = layout(case)
        return {"bytes": 16 * sum(ny * nx for ny, nx, _, _ in items),
                "flops": 9 * sum(ny * nx * t for ny, nx, _, t in items)}
    cells = int(np.prod(shape_of(case)))
    if case["kind"] == "diffuse":  # forward, transposed step and two products per face and step
        nd = case["ndim"]
        return {"bytes": 48 * cells, "flops": cells * case["steps"] * (2 * (4 * nd + 1) + 4 * nd)}
    return {"bytes": 16 * cells, "flops": (2 * n_taps(case["stencil"], case["ndim"]) - 1) * cells * case["steps"]}


# ------------------------------------------------- the same in plain torch


def moved(u, offset, periodic):
    """v[x] = u[x + offset] (zeros from outside when not periodic)."""
    if periodic:
        return torch.roll(u, [-o for o in offset], list(range(u.dim())))
    v = torch.zeros_like(u)
    to = tuple(slice(max(0, -o), max(0, n - max(0, o))) for o, n in zip(offset, u.shape))
    of = tuple(slice(max(0, o), max(0, n + min(0, o))) for o, n in zip(offset, u.shape))
    if all(abs(o) < n for o, n in zip(offset, u.shape)):
        v[to] = u[of]
    return v


def split(u):
    """u as a sum of two halves of 26 bits each (Veltkamp), whose products are exact."""
    c = u * 134217729.0
    high = c - (c - u)
    return high, u - high


def sweep(u, w, periodic, steps):
    """The sum over the taps, step by step, in pairs of 64-bit numbers (value
    and remainder), rounded once at the end: a plain 64-bit sum has rounding
    errors of its own, as large as the ones that it is to show."""
    r = w.shape[0] // 2
    taps = [(tuple(int(i) - r for i in k), torch.tensor(float(w[k]), dtype=torch.float64, device=u.device))
            for k in np.ndindex(*w.shape) if w[k] != 0.0]
    rest = torch.zeros_like(u)
    for _ in range(steps):
        high, low = split(u)
        total, err = torch.zeros_like(u), torch.zeros_like(u)
        for offset, weight in taps:
            wh, wl = split(weight)
            p = weight * moved(u, offset, periodic)
            h, l = moved(high, offset, periodic), moved(low, offset, periodic)
            err += ((wh * h - p) + wh * l + wl * h) + wl * l  # what rounding took from the product
            err += weight * moved(rest, offset, periodic)
            new = total + p
            back = new - total
            err += (total - (new - back)) + (p - back)  # what rounding took from the sum
            total = new
        u = total + err
        rest = err - (u - total)
    return u


def exact(case, seed):
    if case["kind"] == "batch":
        gen, out = generator(seed), []
        for ny, nx, a, t in layout(case):
            u = torch.rand(ny, nx, generator=gen, dtype=torch.float64, device="cuda")
            w = np.array([[0, a, 0], [a, 1 - 4 * a, a], [0, a, 0]])
            out.append(sweep(u, w, case["periodic"], t))
        return out
    if case["kind"] == "const":
        return sweep(field(case["field"], shape_of(case), generator(seed)), weights_of(case), case["periodic"],
                     case["steps"])
    # the chain rule of u' = u + dt * sum over faces of (kappa_i + kappa_n) / 2 * (u_n - u_i), step by step
    u, kappa, lam, dt = diffuse_inputs(case, seed)
    per, nd = case["periodic"], case["ndim"]
    if u.numel() * case["steps"] > 2e9:
        return None
    offsets = [tuple(s if d == e else 0 for e in range(nd)) for d in range(nd) for s in (-1, 1)]
    inside = [moved(torch.ones_like(u), o, per) for o in offsets]  # 0 where the neighbour is a ghost
    # a ghost face has the diffusivity of its own cell and u = 0 outside
    kf = [0.5 * (kappa + moved(kappa, o, per)) * m + kappa * (1 - m) for o, m in zip(offsets, inside)]
    states = []
    for _ in range(case["steps"]):
        states.append(u)
        u = u + dt * sum(k * (moved(u, o, per) - u) for o, k in zip(offsets, kf))
    grad = torch.zeros_like(kappa)
    for v in reversed(states):
        for o, m in zip(offsets, inside):
            dl, dv = lam - moved(lam, o, per), v - moved(v, o, per)
            grad -= 0.5 * dt * dl * dv * (1 + (1 - m))
        lam = lam + dt * sum(k * (moved(lam, o, per) - lam) for o, k in zip(offsets, kf))
    return [u, lam, grad]
