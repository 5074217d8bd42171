"""What the performance of this library is measured on: the calls its users make, from the
smallest to the largest sizes of the repository's own workloads (tests, benchmark, paper).

Every case goes through the package's public functions with inputs resident on the GPU, and a
pass is what a program does once per step: rebuild the cell list and sum over the pairs, one
training step of a kernel model, one prediction, one fit.

Kinds of case and what each stands for:

``velocity``  the paper's velocity update (Sec. 3, Fig. 3): rebuild, the exponential force of
              Eq. 1, ``v += f``.  From a thousand particles (latency) to a million, with the
              neighbour count fixed (~9.4) or growing with the density (over a thousand).
``gauss``     a Gaussian pair sum as a layer under autograd: forward, then the gradients in
              positions and weights.  Uniform points in 2-D, and the clustered 3-D points.
``lj``        molecular dynamics: rebuild and Lennard-Jones energy and forces.  Either through
              autograd with a per-particle upstream gradient (periodic or with walls), or the
              one-call step with packed coordinates and the total energy (large systems).
``step``      a whole time step in place, rebuild included: soft repulsion, then the Brownian
              or the molecular-dynamics integrator.
``sph``       one smoothed-particle-hydrodynamics pass: rebuild, density, pressure, force.
``predict``   the posterior mean of a Gaussian process (or an RBF interpolant) at new points:
              a dense kernel product, one to a few targets in FP32.
``train``     one training step of a dense kernel model: forward, then the gradients in
              points, weights and the length scale, in FP32 or on the tensor cores.
``fit``       the conjugate-gradient solve of a kernel system.

The particles of ``lj`` and ``sph`` sit on a jittered lattice in shuffled order (a liquid has no
overlapping particles); the others are uniform or clustered as in the paper's workloads.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1704_08907_gb300 as ab

DEV = torch.device("cuda", 0)


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the paper's velocity update on a thousand particles, ~9.4 neighbours: all latency
        {"name": "velocity_1k", "kind": "velocity", "dim": 2, "n": 1000, "neighbours": 9.4},
        # Fig. 3's other line, radius fixed as the density grows: ~1235 neighbours a particle
        {"name": "velocity_65k_dense", "kind": "velocity", "dim": 2, "n": 65536,
         "neighbours": 1235.0},
        # the 2-D periodic Gaussian layer of 4096 points (r = 0.03), forward and backward
        {"name": "gauss_2d_4096", "kind": "gauss", "dim": 2, "n": 4096, "neighbours": 11.6,
         "blobs": 0},
        # the clustered layer: 16.7M points in 1024 blobs, forward and backward
        {"name": "gauss_clustered_16M", "kind": "gauss", "dim": 3, "n": 1 << 24,
         "neighbours": 64.0, "blobs": 1024},
        # a mid-size molecular system between two walls, differentiated by autograd
        {"name": "lj_walls_100k", "kind": "lj", "dim": 3, "n": 100003, "neighbours": 33.6,
         "walls": 1, "total": False},
        # the benchmark's molecular-dynamics step: a million particles, packed coordinates
        {"name": "lj_step_1M", "kind": "lj", "dim": 3, "n": 1 << 20, "neighbours": 33.6,
         "walls": 0, "total": True},
        # Brownian dynamics of 4M particles, one axis periodic, one reflecting
        {"name": "brownian_4M", "kind": "step", "dim": 2, "n": 1 << 22, "neighbours": 52.7,
         "walls": 1, "integrator": "brownian"},
        # one SPH pass over a million particles, ~57 neighbours
        {"name": "sph_1M", "kind": "sph", "dim": 3, "n": 1000000, "neighbours": 57.0, "walls": 0},
        # Gaussian-process mean at 2000 new points from 30,000 observations of one target
        {"name": "predict_one_target", "kind": "predict", "m": 2000, "n": 30000, "nrhs": 1,
         "prec": "fp32"},
        # a training step of a 16-output kernel model in FP32 on odd sizes
        {"name": "train_fp32_16", "kind": "train", "m": 5001, "n": 12345, "nrhs": 16,
         "prec": "fp32"},
        # the benchmark's dense operator, forward and backward on the tensor cores
        {"name": "train_bf16x3_65k", "kind": "train", "m": 65536, "n": 65536, "nrhs": 64,
         "prec": "bf16x3"},
        # fitting a Gaussian process to 4096 observations of one target
        {"name": "fit_one_target", "kind": "fit", "n": 4096, "nrhs": 1, "noise": 0.5,
         "prec": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["velocity", "gauss", "lj", "step", "sph", "predict", "train", "fit"])
    if kind == "velocity":
        n = _log(rng, 500, 1 << 20)
        top = min(1235.0, n / 8.0, 8.1e7 / n)
        nb = rng.choice([9.4, math.exp(rng.uniform(math.log(5.0), math.log(max(top, 6.0))))])
        return {"kind": kind, "dim": rng.choice([2, 2, 3]), "n": n, "neighbours": nb}
    if kind == "gauss":
        blobs = rng.choice([0, 0, 256, 1024])
        n = _log(rng, 2000, 1 << 20) if not blobs else _log(rng, 512 * blobs, blobs << 14)
        return {"kind": kind, "dim": 3 if blobs else rng.choice([2, 3]), "n": n,
                "neighbours": rng.uniform(10.0, 64.0), "blobs": blobs}
    if kind == "lj":
        total = rng.random() < 0.5
        n = _log(rng, 1 << 19, 1 << 21) if total else _log(rng, 2000, 1 << 19)
        return {"kind": kind, "dim": 3 if total else rng.choice([2, 3]), "n": n,
                "neighbours": rng.uniform(20.0, 40.0), "walls": 0 if total else rng.choice([0, 1, 2]),
                "total": total}
    if kind == "step":
        return {"kind": kind, "dim": rng.choice([2, 3]), "n": _log(rng, 2000, 1 << 22),
                "neighbours": rng.uniform(10.0, 53.0), "walls": rng.choice([0, 1, 2]),
                "integrator": rng.choice(["brownian", "molecular"])}
    if kind == "sph":
        return {"kind": kind, "dim": rng.choice([2, 3]), "n": _log(rng, 5000, 1 << 20),
                "neighbours": rng.uniform(20.0, 60.0), "walls": rng.choice([0, 1])}
    if kind == "predict":
        prec = rng.choice(["fp32", "fp32", "fp32", "bf16x3", "tf32x3", "bf16", "tf32"])
        return {"kind": kind, "m": _log(rng, 100, 30000), "n": _log(rng, 1000, 60000),
                "nrhs": 64 if prec != "fp32" else rng.choice([1, 1, 2, 3, 5, 8, 17, 64]),
                "prec": prec}
    if kind == "train":
        prec = rng.choice(["fp32", "fp32", "bf16x3", "tf32x3"])
        return {"kind": kind, "m": _log(rng, 500, 20000), "n": _log(rng, 500, 20000),
                "nrhs": 64 if prec != "fp32" else rng.choice([1, 1, 4, 10, 16, 33, 64]),
                "prec": prec}
    prec = rng.choice(["fp32", "fp32", "fp32", "bf16x3"])
    return {"kind": kind, "n": _log(rng, 500, 4096),
            "nrhs": 64 if prec != "fp32" else rng.choice([1, 1, 2, 4]),
            "noise": rng.uniform(0.3, 1.0), "prec": prec}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(1704089 + seed)


def _pack4(x):
    out = torch.zeros((x.shape[0], 4), dtype=torch.float32, device=DEV)
    out[:, :x.shape[1]] = x
    out[out >= 1.0] = 0.0
    return out


def _uniform(n, dim, g):
    return _pack4(torch.rand((n, dim), generator=g, device=DEV))


def _blobs(n, blobs, g):
    """Points in equal Gaussian blobs of standard deviation 0.01, wrapped into the unit cube."""
    centres = torch.rand((blobs, 3), generator=g, device=DEV)
    x = centres[torch.arange(n, device=DEV) % blobs]
    x = x + 0.01 * torch.randn((n, 3), generator=g, device=DEV)
    return _pack4(x - torch.floor(x))


def _liquid(n, dim, g):
    """A jittered lattice with a few vacancies, in shuffled order."""
    side = math.ceil(n ** (1.0 / dim) - 1e-9)
    sites = torch.randperm(side ** dim, generator=g, device=DEV)[:n]
    x = torch.stack([torch.div(sites, side ** k, rounding_mode="floor") % side for k in range(dim)], 1)
    jitter = 0.2 * (torch.rand((n, dim), generator=g, device=DEV) - 0.5)
    return _pack4((x + 0.5 + jitter) / side)


def _radius(case):
    """Cut-off with the wanted mean number of neighbours in the unit box."""
    n, nb, dim = case["n"], case["neighbours"], case["dim"]
    if case.get("blobs"):
        # density seen by a point of its own blob, averaged: (2 sqrt(pi) sd)^-3 a point
        rho = n / case["blobs"] / (2.0 * math.sqrt(math.pi) * 0.01) ** 3 + n
    else:
        rho = float(n)
    return math.sqrt(nb / (math.pi * rho)) if dim == 2 else (nb * 0.75 / (math.pi * rho)) ** (1 / 3)


def _periodic(case):
    walls = min(case.get("walls", 0), case["dim"])
    return [1] * (case["dim"] - walls) + [0] * walls


def _dense_inputs(case, seed):
    """Points in the unit cube; smooth targets with noise; residuals for the backward pass."""
    g = _gen(seed)
    m, n, q = case.get("m", case["n"]), case["n"], case["nrhs"]
    X = _uniform(m, 3, g)
    Y = _uniform(n, 3, g)
    W = torch.randn((n, q), generator=g, device=DEV)
    G = torch.randn((m, q), generator=g, device=DEV)
    return X, Y, W, G


S_DENSE = 50.0      # 1 / (2 l^2), length scale l = 0.1


def prepare(case, seed):
    k = case["kind"]
    st = {"case": case, "ctx": ab.ab_create()}
    if k in ("predict", "train"):
        st["X"], st["Y"], st["W"], st["G"] = _dense_inputs(case, seed)
        if k == "train":
            st["s"] = torch.tensor(S_DENSE, dtype=torch.float32, device=DEV, requires_grad=True)
            for v in "XYW":
                st[v].requires_grad_(True)
        return st
    g = _gen(seed)
    if k == "fit":
        n, q = case["n"], case["nrhs"]
        st["X"] = _uniform(n, 3, g)
        f = torch.sin(2.0 * math.pi * st["X"][:, :1] + torch.arange(q, device=DEV)[None, :])
        st["B"] = (f * torch.cos(3.0 * st["X"][:, 1:2])
                   + case["noise"] * torch.randn((n, q), generator=g, device=DEV)).float().contiguous()
        return st
    n, dim = case["n"], case["dim"]
    r = _radius(case)
    st["dom"] = ab.Domain(dim, _periodic(case), r)
    if k == "velocity":
        st["pos"] = _uniform(n, dim, g)
        st["vel"] = torch.zeros((n, 4), dtype=torch.float32, device=DEV)
        st["f"] = torch.empty((n, 4), dtype=torch.float32, device=DEV)
        st["prm"] = ab.OpParams(c=1e-3)
    elif k == "gauss":
        st["pos"] = _blobs(n, case["blobs"], g) if case["blobs"] else _uniform(n, dim, g)
        st["w"] = torch.randn(n, generator=g, device=DEV)
        st["g"] = torch.randn(n, generator=g, device=DEV)
        st["s"] = (3.0 / r) ** 2
        st["pos"].requires_grad_(True)
        st["w"].requires_grad_(True)
    elif k == "lj":
        st["pos"] = _liquid(n, dim, g)
        st["sigma"] = 1.0 / math.ceil(n ** (1.0 / dim) - 1e-9)
        if case["total"]:
            st["pos"] = st["pos"][:, :dim].contiguous()
            st["E"] = torch.empty(n, dtype=torch.float32, device=DEV)
            st["F"] = torch.empty((n, dim), dtype=torch.float32, device=DEV)
            st["energy"] = torch.empty((), dtype=torch.float64, device=DEV)
        else:
            st["pos"].requires_grad_(True)
            st["g"] = 0.5 + torch.rand(n, generator=g, device=DEV)
    elif k == "step":
        st["pos"] = _uniform(n, dim, g)
        st["vel"] = torch.zeros((n, 4), dtype=torch.float32, device=DEV)
        st["f"] = torch.empty((n, 4), dtype=torch.float32, device=DEV)
        st["prm"] = ab.OpParams(k=1e4 if case["integrator"] == "brownian" else 1.0)
        st["seed"], st["step"] = seed, 0
    elif k == "sph":
        st["pos"] = _liquid(n, dim, g)
        st["mass"] = (0.9 + 0.2 * torch.rand(n, generator=g, device=DEV)) / n
        st["prm"] = ab.OpParams()
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
DT_BD, D_BD = 1e-5, 1e-2      # the Brownian workload's time step and diffusion constant
DT_MD = 1e-3


def run(st):
    case, ctx = st["case"], st["ctx"]
    k = case["kind"]
    if k == "velocity":
        ab.ab_build(ctx, st["dom"], st["pos"])
        f = ab.ab_pair_sum(ctx, "expf", st["prm"], out=st["f"])
        st["vel"].add_(f)
        return {"force": f, "vel": st["vel"]}
    if k == "gauss":
        y = ab.GaussPairSum.apply(st["pos"], st["w"], st["s"], ctx, st["dom"])
        gp, gw = torch.autograd.grad(y, (st["pos"], st["w"]), st["g"])
        return {"y": y, "grad_pos": gp, "grad_w": gw}
    if k == "lj":
        if case["total"]:
            E, F, energy = ab.lj_energy_forces(ctx, st["dom"], st["pos"], 1.0, st["sigma"],
                                               E=st["E"], F=st["F"], energy=st["energy"])
            return {"E": E, "grad_pos": F, "energy": energy}
        E = ab.LJEnergy.apply(st["pos"], ctx, st["dom"], 1.0, st["sigma"])
        (gp,) = torch.autograd.grad(E, (st["pos"],), st["g"])
        return {"E": E, "grad_pos": gp}
    if k == "step":
        ab.ab_build(ctx, st["dom"], st["pos"])
        f = ab.ab_pair_sum(ctx, "soft", st["prm"], out=st["f"])
        st["step"] += 1
        if case["integrator"] == "brownian":
            ab.ab_bd_step(ctx, st["dom"], st["pos"], f, DT_BD, D_BD, st["seed"], st["step"])
            return {"pos": st["pos"], "force": f}
        ab.ab_md_step(ctx, st["dom"], st["pos"], st["vel"], f, DT_MD)
        return {"pos": st["pos"], "vel": st["vel"], "force": f}
    if k == "sph":
        ab.ab_build(ctx, st["dom"], st["pos"])
        rho = ab.ab_pair_sum(ctx, "sph_density", st["prm"], w=st["mass"])
        ma = torch.stack([st["mass"], torch.reciprocal(rho)], 1)     # P = rho: A = P / rho^2
        acc = ab.ab_pair_sum(ctx, "sph_force", st["prm"], w=ma)
        return {"rho": rho, "acc": acc}
    if k == "predict":
        return ab.ab_kernel_matvec(ctx, st["X"], st["Y"], st["W"], S_DENSE, case["prec"])
    if k == "train":
        out = ab.KernelMatvec.apply(st["X"], st["Y"], st["W"], st["s"], ctx, case["prec"])
        gX, gY, gW, gs = torch.autograd.grad(out, (st["X"], st["Y"], st["W"], st["s"]), st["G"])
        return {"out": out, "grad_X": gX, "grad_Y": gY, "grad_W": gW, "grad_s": gs}
    W, iters, _ = ab.ab_kernel_solve(ctx, st["X"], st["B"], S_DENSE, case["noise"] ** 2,
                                     case["prec"], tol=1e-4, max_iter=1000)
    return {"W": W, "iters": iters}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Inputs read once and outputs written once; the arithmetic of the accepted pairs (or of
    all pairs of a dense operator).  An exponential or a reciprocal counts as one operation."""
    k = case["kind"]
    if k in ("predict", "train"):
        m, n, q = case["m"], case["n"], case["nrhs"]
        fwd = m * n * (9.0 + 2.0 * q)
        if k == "predict":
            return {"bytes": 16.0 * (m + n) + 4.0 * q * (m + n), "flops": fwd}
        # dW: the forward's work again; dX, dY, ds: G_i . W_j, then 8 operations for each
        return {"bytes": 2 * 16.0 * (m + n) + 4.0 * q * (2 * m + 2 * n),
                "flops": 2 * fwd + m * n * (2.0 * q + 25.0)}
    if k == "fit":
        n, q = case["n"], case["nrhs"]
        iters = 40          # an order of magnitude: it depends on the data
        return {"bytes": 16.0 * n + 8.0 * q * n, "flops": iters * n * n * (9.0 + 2.0 * q)}
    n, dim, nb = case["n"], case["dim"], case["neighbours"]
    pairs = n * nb
    pos, vec = 16.0, 16.0
    if k == "velocity":
        return {"bytes": n * (pos + vec + 2 * vec), "flops": pairs * (3 * dim + 5 + 2 * dim)}
    if k == "gauss":
        return {"bytes": n * (pos + 4 + 4 + 4 + vec + 4), "flops": pairs * (3 * dim + 4 + 2 * dim + 7)}
    if k == "lj":
        g = 4.0 * dim if case["total"] else 16.0
        return {"bytes": n * (g + 4 + g + (0 if case["total"] else 4)),
                "flops": pairs * (3 * dim + 10 + 2 * dim)}
    if k == "step":
        moved = 2 * pos + vec + (0 if case["integrator"] == "brownian" else 2 * vec)
        return {"bytes": n * moved, "flops": pairs * (3 * dim + 7 + 2 * dim) + n * 100.0}
    return {"bytes": n * (pos + 4 + 4 + 4 + 8 + vec), "flops": pairs * (2 * 3 * dim + 9 + 9 + 2 * dim)}


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _pairs(pos, case, r):
    """Blocks (i, j, dx, d2) of all ordered neighbour pairs.  The relation is the library's FP32
    rule (minimum image, squares and sums each rounded); separations are in 64 bits."""
    n, dim = case["n"], case["dim"]
    x = pos[:, :dim].contiguous()
    per = _periodic(case)
    r32 = torch.tensor(r, dtype=torch.float32, device=DEV)
    r2 = r32 * r32

    def accepted(i, j):
        d = x[j] - x[i]
        wide = x[j].double() - x[i].double()
        for a in range(dim):
            if per[a]:
                c = d[:, a]
                up, down = c > 0.5, c < -0.5
                d[:, a] = torch.where(up, c - 1.0, torch.where(down, c + 1.0, c))
                wide[:, a] += down.double() - up.double()
        q = d * d
        d2 = q[:, 0] + q[:, 1]
        if dim == 3:
            d2 = d2 + q[:, 2]
        keep = (d2 < r2) & (i != j)
        i, j, wide = i[keep], j[keep], wide[keep]
        return i, j, wide, (wide * wide).sum(1)

    cells = int(math.floor(1.0 / (r * 1.0001)))
    if cells < 4 or n <= 4096:
        rows = max(1, (1 << 25) // n)
        for a in range(0, n, rows):
            b = min(n, a + rows)
            i = torch.arange(a, b, device=DEV).repeat_interleave(n)
            yield accepted(i, torch.arange(n, device=DEV).repeat(b - a))
        return
    cells = min(cells, 2000 if dim == 2 else 400)
    c = (x.double() * cells).floor().long().clamp_(0, cells - 1)
    key = c[:, 0]
    for a in range(1, dim):
        key = key * cells + c[:, a]
    skey, order = torch.sort(key)
    every = torch.arange(n, device=DEV)
    for o in range(3 ** dim):
        t, live, nkey = o, torch.ones(n, dtype=torch.bool, device=DEV), torch.zeros_like(key)
        for a in range(dim):
            ca = c[:, a] + (t % 3 - 1)
            t //= 3
            if per[a]:
                ca = ca % cells
            else:
                live &= (ca >= 0) & (ca < cells)
            nkey = nkey * cells + ca
        i = every[live]
        lo = torch.searchsorted(skey, nkey[live])
        count = torch.searchsorted(skey, nkey[live], right=True) - lo
        # in chunks of at most 2^25 candidates
        ends = torch.cumsum(count, 0)
        a = 0
        while a < i.numel():
            base = int(ends[a - 1]) if a else 0
            b = max(a + 1, int(torch.searchsorted(ends, torch.tensor(base + (1 << 25), device=DEV),
                                                  right=True)))
            ii = i[a:b].repeat_interleave(count[a:b])
            if ii.numel():
                first = (ends[a:b] - count[a:b] - base).repeat_interleave(count[a:b])
                at = torch.arange(ii.numel(), device=DEV) - first
                yield accepted(ii, order[lo[a:b].repeat_interleave(count[a:b]) + at])
            a = b


def _add(to, i, v):
    to.index_add_(0, i, v)


def _exact_pairs(case, st):
    k, n, dim = case["kind"], case["n"], case["dim"]
    r = float(np.float32(_radius(case)))
    pos = st["pos"].detach()
    if pos.shape[1] != 4:
        pos = _pack4(pos)
    f64 = dict(dtype=torch.float64, device=DEV)
    vec = torch.zeros((n, 4), **f64)
    y = torch.zeros(n, **f64)
    if k == "velocity":
        c = float(np.float32(1e-3))
        for i, j, dx, d2 in _pairs(pos, case, r):
            d = torch.sqrt(d2)
            mag = torch.where(d > 0, -c * torch.exp(-d) / d.clamp_min(1e-300), 0.0 * d)
            _add(vec[:, :dim], i, mag[:, None] * dx)
        return {"force": vec, "vel": st["vel"].double() + vec}
    if k == "gauss":
        s = float(np.float32(st["s"]))
        w, g, gw = st["w"].detach().double(), st["g"].double(), torch.zeros(n, **f64)
        for i, j, dx, d2 in _pairs(pos, case, r):
            e = torch.exp(-s * d2)
            _add(y, i, w[j] * e)
            _add(gw, i, g[j] * e)
            _add(vec[:, :dim], i, ((g[i] * w[j] + g[j] * w[i]) * (2.0 * s) * e)[:, None] * dx)
        return {"y": y, "grad_pos": vec, "grad_w": gw}
    if k == "lj":
        sig2 = float(np.float32(st["sigma"])) ** 2
        g = torch.ones(n, **f64) if case["total"] else st["g"].double()
        for i, j, dx, d2 in _pairs(pos, case, r):
            s6 = (sig2 / d2) ** 3
            _add(y, i, 0.5 * (s6 * s6 - s6))
            _add(vec[:, :dim], i, (0.5 * (g[i] + g[j]) * (12.0 * s6 * s6 - 6.0 * s6) / d2)[:, None] * dx)
        if case["total"]:
            return {"E": y, "grad_pos": vec[:, :dim].contiguous(), "energy": y.sum()}
        return {"E": y, "grad_pos": vec}
    if k == "sph":
        pi = math.pi
        a = 21.0 / (2.0 * pi * r ** 3) if dim == 3 else 7.0 / (pi * r * r)
        m = st["mass"].double()
        y += m * a
        for i, j, dx, d2 in _pairs(pos, case, r):
            q = torch.sqrt(d2) / r
            _add(y, i, m[j] * a * (1.0 - q).clamp_min(0.0) ** 4 * (1.0 + 4.0 * q))
        A = 1.0 / y
        for i, j, dx, d2 in _pairs(pos, case, r):
            t = (1.0 - torch.sqrt(d2) / r).clamp_min(0.0)
            _add(vec[:, :dim], i, (m[j] * (A[i] + A[j]) * (-20.0 * a / (r * r)) * t ** 3)[:, None] * dx)
        return {"rho": y, "acc": vec}
    # step: soft repulsion, then the integrator
    kk = 1e4 if case["integrator"] == "brownian" else 1.0
    for i, j, dx, d2 in _pairs(pos, case, r):
        d = torch.sqrt(d2)
        mag = torch.where(d > 0, -kk * (r - d) / d.clamp_min(1e-300), 0.0 * d)
        _add(vec[:, :dim], i, mag[:, None] * dx)
    x = pos.double()
    vel = st["vel"].double()
    if case["integrator"] == "brownian":
        dt, D = float(np.float32(DT_BD)), float(np.float32(D_BD))
        raw = np.random.Philox(key=st["seed"], counter=(1 << 64) - 1).random_raw(4 * n).reshape(n, 4)
        u = torch.from_numpy(((raw >> np.uint64(40)).astype(np.float64) + 1.0) * 2.0 ** -24).to(DEV)
        rad = torch.sqrt(-2.0 * torch.log(u[:, 0::2]))
        z = torch.stack([rad[:, 0] * torch.cos(2 * math.pi * u[:, 1]),
                         rad[:, 0] * torch.sin(2 * math.pi * u[:, 1]),
                         rad[:, 1] * torch.cos(2 * math.pi * u[:, 3])], 1)
        move = dt * vec[:, :dim] + math.sqrt(2.0 * D * dt) * z[:, :dim]
    else:
        dt = float(np.float32(DT_MD))
        vel[:, :dim] += dt * vec[:, :dim]
        move = dt * vel[:, :dim]
    per = _periodic(case)
    for a in range(dim):
        p = x[:, a] + move[:, a]
        if per[a]:
            p = p - torch.floor(p)
            p = torch.where(p.float() >= 1.0, p - p, p)
        else:
            low, high = p < 0.0, p > 1.0
            p = torch.where(low, -p, torch.where(high, 2.0 - p, p))
            if case["integrator"] != "brownian":
                vel[:, a] = torch.where(low | high, -vel[:, a], vel[:, a])
        x[:, a] = p
    if case["integrator"] == "brownian":
        return {"pos": x, "force": vec}
    return {"pos": x, "vel": vel, "force": vec}


def _exact_dense(case, st):
    X, Y, W, G = (st[v].detach().double() for v in "XYWG")
    X, Y = X[:, :3], Y[:, :3]
    train = case["kind"] == "train"
    out = torch.empty((X.shape[0], W.shape[1]), dtype=torch.float64, device=DEV)
    gX, gY = torch.zeros((X.shape[0], 4), dtype=torch.float64, device=DEV), torch.zeros(
        (Y.shape[0], 4), dtype=torch.float64, device=DEV)
    gW = torch.zeros_like(W)
    gs = torch.zeros((), dtype=torch.float64, device=DEV)
    s = S_DENSE
    rows = max(1, (1 << 27) // Y.shape[0])
    for a in range(0, X.shape[0], rows):
        x = X[a:a + rows]
        d2 = sum((x[:, k, None] - Y[None, :, k]) ** 2 for k in range(3))
        K = torch.exp(-s * d2)
        out[a:a + rows] = K @ W
        if train:
            g = G[a:a + rows]
            gW += K.T @ g
            A = K * (g @ W.T)
            gs -= (A * d2).sum()
            gX[a:a + rows, :3] = -2.0 * s * (x * A.sum(1, keepdim=True) - A @ Y)
            gY[:, :3] += 2.0 * s * (A.T @ x - Y * A.sum(0)[:, None])
    if not train:
        return out
    return {"out": out, "grad_X": gX, "grad_Y": gY, "grad_W": gW, "grad_s": gs}


def exact(case, seed):
    st = prepare(case, seed)
    k = case["kind"]
    if k in ("predict", "train"):
        return _exact_dense(case, st)
    if k == "fit":
        # the solution that the iteration tends to (its own error is the stopping tolerance's)
        X = st["X"][:, :3].double()
        d2 = sum((X[:, a, None] - X[None, :, a]) ** 2 for a in range(3))
        K = torch.exp(-S_DENSE * d2)
        K.diagonal().add_(case["noise"] ** 2)
        return {"W": torch.linalg.solve(K, st["B"].double()), "iters": None}
    return _exact_pairs(case, st)
