"""The solves this library is used for, as cases to be timed.

A case is a plain dict.  ``kind`` says which entry point a user calls:

  solve   Solver(...)(f, u): one domain, one precision, device buffers
  multi   lgf_plan_create_multi + lgf_solve: equal small requests folded into one plan
  batch   BatchSolver: many uneven problems of two block sizes, one CUDA graph
  conv    lgf_conv_blocks: every block its own one-block domain
  host    lgf_solve_host_pipelined: a sequence of host inputs, copies overlapped

Domains: ``box`` (all nb^3 blocks), ``sphere`` / ``shell`` (blocks whose centre
lies in the ball, or between half and all of its radius) and ``tori`` (the
blocks where a sum of random Gaussian tori exceeds 1e-6 of its maximum).
Sources are made on the GPU from the seed: tori with 5% multiplicative noise
(non-negative, smooth; the vorticity-like fields of the method's experiments),
or noise in (-1, 1) for the convolution of isolated blocks.

``exact`` is the lattice convolution u = G * f itself, in 64 bits by one
zero-padded FFT over the bounding box, with G from its Bessel integral.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1402_6081_gb300 as lgf

_PREC = {"fp32": (lgf.LGF_FP32, torch.float32), "fp64": (lgf.LGF_FP64, torch.float64)}


# ---- the cases ----

def listed():
    return [
        # the two-level 32^3 Gaussian-sized box, 8^3 blocks, order 6: the smallest request, all launches
        {"name": "box_32_nb8", "kind": "solve", "domain": "box", "n_b": 8, "nb": 4, "order": 6, "prec": "fp32"},
        # eight pending requests of one small shape folded into one plan, as the server does
        {"name": "fold_8x24_nb8", "kind": "multi", "domain": "box", "n_b": 8, "nb": 3, "copies": 8, "order": 8,
         "prec": "fp32"},
        # the single-solve workload of the benchmark, in the serving precision ...
        {"name": "box_128_nb16", "kind": "solve", "domain": "box", "n_b": 16, "nb": 8, "order": 8, "prec": "fp32"},
        # ... and in the precision of the error experiments
        {"name": "box_128_nb16_fp64", "kind": "solve", "domain": "box", "n_b": 16, "nb": 8, "order": 8,
         "prec": "fp64"},
        # the same box on small blocks: a tree of four levels, many small transforms
        {"name": "box_128_nb8", "kind": "solve", "domain": "box", "n_b": 8, "nb": 16, "order": 8, "prec": "fp32"},
        # the largest request of the Poisson stream (2^24 points)
        {"name": "box_256_nb16", "kind": "solve", "domain": "box", "n_b": 16, "nb": 16, "order": 8, "prec": "fp32"},
        # the 512^3 irregular domain: five levels, a fifth of the box occupied
        {"name": "tori_512_nb16", "kind": "solve", "domain": "tori", "n_b": 16, "nb": 32, "order": 8,
         "prec": "fp32", "domain_seed": 2},
        # the error experiments: a ball, order 9, 64 bits, a block size that is no power of two
        {"name": "sphere_96_nb12_fp64", "kind": "solve", "domain": "sphere", "n_b": 12, "nb": 8, "order": 9,
         "prec": "fp64"},
        # large blocks (the upper end of the error experiments' range)
        {"name": "box_144_nb24", "kind": "solve", "domain": "box", "n_b": 24, "nb": 6, "order": 8, "prec": "fp32"},
        # batched serving of uneven problems
        {"name": "batch_24_uneven", "kind": "batch", "problems": 24, "domain_seed": 3, "prec": "fp32"},
        # the paper's "FFT Conv." special case: 512 isolated blocks
        {"name": "conv_512_nb16", "kind": "conv", "blocks": 512, "n_b": 16, "prec": "fp32"},
        # end to end from pinned host memory: a stream of inputs through one plan
        {"name": "host_128_nb16", "kind": "host", "domain": "box", "n_b": 16, "nb": 8, "order": 8, "prec": "fp32",
         "steps": 4},
    ]


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["multi", "batch", "conv", "host"])
    prec = "fp32" if rng.random() < 0.7 else "fp64"
    if kind == "conv":
        n_b = rng.choice([4, 8, 16])
        points = math.exp(rng.uniform(math.log(2.0 ** 14), math.log(2.0 ** 23)))
        return {"kind": kind, "blocks": max(1, int(points / n_b ** 3)), "n_b": n_b, "prec": prec}
    if kind == "batch":
        return {"kind": kind, "problems": rng.randint(3, 32), "domain_seed": rng.randrange(10 ** 6), "prec": "fp32"}
    if kind == "multi":
        n_b = rng.choice([4, 6, 8, 8, 16])
        return {"kind": kind, "domain": rng.choice(["box", "sphere"]), "n_b": n_b,
                "nb": rng.randint(2, max(2, 48 // n_b)), "copies": rng.randint(2, 9), "order": min(8, n_b),
                "prec": prec}
    # points of the bounding box, over the logarithm of the range; 64 bits up to 128^3
    top = 21.0 if prec == "fp64" else 24.0 if kind == "solve" else 22.0
    n_b = rng.choice([16] * 5 + [8] * 4 + [4, 6, 10, 12, 14, 18, 20, 24, 28, 32])
    if n_b <= 6 or n_b >= 18:
        top = min(top, 21.0)
    side = 2.0 ** (rng.uniform(13.0, top) / 3.0)
    nb = max(1, round(side / n_b))
    domain = rng.choice(["box", "box", "sphere", "shell", "tori"]) if nb > 2 else "box"
    order = rng.choice([o for o in (4, 6, 7, 8, 8, 8, 9) if o <= n_b])
    c = {"kind": kind, "domain": domain, "n_b": n_b, "nb": nb, "order": order, "prec": prec}
    if domain == "tori":
        c["domain_seed"] = rng.randrange(10 ** 6)
    if kind == "host":
        c["steps"] = rng.randint(1, 6)
    return c


# ---- domains and sources ----

def _levels(nb: int) -> int:
    return max(1, math.ceil(math.log2(max(nb, 1))))


def _box(nb: int):
    z, y, x = np.meshgrid(np.arange(nb), np.arange(nb), np.arange(nb), indexing="ij")
    return np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1).astype(np.int32)


def _tori(rng, side: float, count: int):
    """Centre, normal, radius, core width, amplitude of random tori in a box."""
    out = []
    for _ in range(count):
        centre = [rng.uniform(side / 4, 3 * side / 4) for _ in range(3)]
        n = [rng.gauss(0, 1) for _ in range(3)]
        r = math.sqrt(sum(v * v for v in n)) or 1.0
        radius = side * math.exp(rng.uniform(math.log(0.04), math.log(0.235)))
        out.append((centre, [v / r for v in n], radius, side * rng.uniform(0.012, 0.031), rng.uniform(0.5, 1.0)))
    return out


def _field(blocks, n_b: int, tori):
    """Sum of the tori at the points of the blocks, (n, n_b, n_b, n_b) in 64 bits, on the GPU."""
    b = torch.as_tensor(blocks, device="cuda", dtype=torch.float64) * n_b
    r = torch.arange(n_b, device="cuda", dtype=torch.float64)
    f = torch.zeros((len(blocks), n_b, n_b, n_b), device="cuda", dtype=torch.float64)
    step = max(1, (1 << 25) // n_b ** 3)
    for a in range(0, len(blocks), step):
        x = b[a:a + step, 0, None, None, None] + r[None, None, None, :]
        y = b[a:a + step, 1, None, None, None] + r[None, None, :, None]
        z = b[a:a + step, 2, None, None, None] + r[None, :, None, None]
        for c, n, radius, sigma, amp in tori:
            vx, vy, vz = x - c[0], y - c[1], z - c[2]
            ax = vx * n[0] + vy * n[1] + vz * n[2]
            rho = ((vx - ax * n[0]) ** 2 + (vy - ax * n[1]) ** 2 + (vz - ax * n[2]) ** 2).sqrt()
            f[a:a + step] += amp * torch.exp(-((rho - radius) ** 2 + ax ** 2) / (2 * sigma ** 2))
    return f


def _domain(case):
    """Blocks of a case's domain and the tori that its sources are made of."""
    n_b, nb, side = case["n_b"], case["nb"], case["n_b"] * case["nb"]
    blocks = _box(nb)
    tori = [([(side - 1) / 2] * 3, [0.0, 0.0, 1.0], 0.3 * side, max(1.5, 0.05 * side), 1.0)]
    if case["domain"] in ("sphere", "shell"):
        r = np.sqrt((((blocks + 0.5) - nb / 2.0) ** 2).sum(axis=1)) / (nb / 2.0)
        blocks = blocks[(r <= 1.0) & ((r >= 0.5) | (case["domain"] == "sphere"))]
    elif case["domain"] == "tori":
        tori = _tori(random.Random(case["domain_seed"]), float(side), 12)
        top = torch.cat([_field(blocks[a:a + 8192], n_b, tori).amax(dim=(1, 2, 3))
                         for a in range(0, len(blocks), 8192)])
        blocks = blocks[(top > 1e-6 * top.max()).cpu().numpy()]
    return np.ascontiguousarray(blocks), tori


def _source(blocks, n_b: int, tori, seed: int):
    """The tori with 5% multiplicative noise of this seed."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    f = _field(blocks, n_b, tori)
    return f.mul_(1.0 + 0.05 * (2.0 * torch.rand(f.shape, generator=g, device="cuda", dtype=torch.float64) - 1.0))


def _batch(case):
    """(blocks, n_b, n_levels, tori) of the problems: boxes of 32 to 160 points, 8^3 or 16^3 blocks,
    the blocks that one to four tori reach."""
    rng = random.Random(case["domain_seed"])
    out = []
    for _ in range(case["problems"]):
        n_b = rng.choice([8, 16])
        nb = max(2, round(math.exp(rng.uniform(math.log(32.0), math.log(160.0))) / n_b))
        side = float(nb * n_b)
        tori = [(c, n, r, max(2.0, 2.0 * s), a) for c, n, r, s, a in _tori(rng, side, rng.randint(1, 4))]
        blocks = _box(nb)
        top = _field(blocks, n_b, tori).amax(dim=(1, 2, 3))
        out.append((blocks[(top > 1e-6 * top.max()).cpu().numpy()], n_b, _levels(nb), tori))
    return out


def _sources(case, seed: int):
    """The case's source fields in 64 bits: a list, one per problem (host: one per step)."""
    if case["kind"] == "conv":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        shape = (case["blocks"],) + (case["n_b"],) * 3
        return [2.0 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 1.0]
    if case["kind"] == "batch":
        return [_source(b, n_b, tori, 1000 * seed + i) for i, (b, n_b, _, tori) in enumerate(_batch(case))]
    blocks, tori = _domain(case)
    n = case.get("copies", case.get("steps", 1))
    return [_source(blocks, case["n_b"], tori, 1000 * seed + i) for i in range(n)]


# ---- what is timed ----

class _Plan:
    """A plan handle that is given back with the state."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        lgf.lgf_destroy(self.handle)


def prepare(case, seed):
    prec, dt = _PREC[case["prec"]]
    f = [x.to(dt) for x in _sources(case, seed)]
    kind = case["kind"]
    if kind == "conv":
        return {"kind": kind, "f": f[0], "u": torch.empty_like(f[0]), "n": case["blocks"], "n_b": case["n_b"],
                "prec": prec}
    if kind == "batch":
        s = lgf.BatchSolver([(b, n_b, levels, 8) for b, n_b, levels, _ in _batch(case)], prec, use_graph=1)
        s.set_sources(f)
        return {"kind": kind, "solver": s, "u": [s.u_view(i) for i in range(len(f))]}
    blocks, _ = _domain(case)
    n_b, levels, order = case["n_b"], _levels(case["nb"]), case["order"]
    if kind == "multi":
        n = case["copies"]
        plan = _Plan(lgf.lgf_plan_create_multi([blocks] * n, n_b, [levels] * n, order, prec))
        f = torch.stack(f)
        return {"kind": kind, "plan": plan, "f": f, "u": torch.empty_like(f)}
    if kind == "host":
        s = lgf.Solver(blocks, n_b, levels, order, prec)
        f = [x.cpu().pin_memory() for x in f]
        return {"kind": kind, "solver": s, "f": f, "u": [torch.empty_like(x).pin_memory() for x in f]}
    return {"kind": kind, "solver": lgf.Solver(blocks, n_b, levels, order, prec), "f": f[0],
            "u": torch.empty_like(f[0])}


def run(state):
    kind = state["kind"]
    if kind == "solve":
        return state["solver"](state["f"], state["u"])
    if kind == "multi":
        lgf.lgf_solve(state["plan"].handle, state["f"], state["u"])
    elif kind == "batch":
        state["solver"]()
    elif kind == "conv":
        lgf.lgf_conv_blocks(state["f"], state["u"], state["n"], state["n_b"], state["prec"])
    else:
        lgf.lgf_solve_host_pipelined(state["solver"].plan, state["f"], state["u"])
    return state["u"]


def work(case):
    """Every input value read and every output value written once; the real transforms of every block,
    padded to twice its edge, both ways, and one complex product per frequency."""
    size = 4 if case["prec"] == "fp32" else 8
    if case["kind"] == "conv":
        parts = [(case["blocks"], case["n_b"])]
    elif case["kind"] == "batch":
        parts = [(len(b), n_b) for b, n_b, _, _ in _batch(case)]
    else:
        parts = [(len(_domain(case)[0]) * case.get("copies", case.get("steps", 1)), case["n_b"])]
    nbytes = flops = 0.0
    for n, n_b in parts:
        padded = (2.0 * n_b) ** 3
        nbytes += 2.0 * size * n * n_b ** 3
        flops += n * (2 * 2.5 * padded * math.log2(padded) + 8 * padded / 2)
    return {"bytes": nbytes, "flops": flops}


# ---- the lattice convolution in 64 bits ----

def _green(n: int):
    """-G(a, b, c) for 0 <= a, b, c <= n: the integral over t of the product of e^(-2t) I_a(2t) and its likes.
    Gauss-Legendre on dyadic panels up to t1, the Bessel functions by the trapezoidal rule of their own
    integral; beyond t1 = 2^12 n^2 the first terms of the large-argument expansion."""
    x, w = (torch.from_numpy(v).cuda() for v in np.polynomial.legendre.leggauss(24))
    top = math.ceil(12 + 2 * math.log2(max(n, 2)))
    edges = [0.0] + [2.0 ** e for e in range(-6, top + 1)]
    rows, weights = [], []
    for a, b in zip(edges[:-1], edges[1:]):
        t = 0.5 * (b - a) * x + 0.5 * (a + b)
        m = 1 << math.ceil(math.log2(2 * n + 64 + 26 * math.sqrt(b)))
        s = torch.sin(torch.arange(m, device="cuda", dtype=torch.float64) * (math.pi / m)) ** 2
        rows.append(torch.fft.rfft(torch.exp(-4.0 * t[:, None] * s[None, :]), dim=1).real[:, :n + 1] / m)
        weights.append(0.5 * (b - a) * w)
    r, w = torch.cat(rows), torch.cat(weights)
    g = ((r * w[:, None])[:, :, None] * r[:, None, :]).reshape(len(r), -1).T @ r
    k = torch.arange(n + 1, device="cuda", dtype=torch.float64) ** 2
    s1 = k[:, None, None] + k[None, :, None] + k[None, None, :]
    t1 = edges[-1]
    # e^(-2t) I_k(2t) = (4 pi t)^(-1/2) (1 - (4 k^2 - 1) / (16 t) + (4 k^2 - 1)(4 k^2 - 9) / (512 t^2) ...)
    p = -(4.0 * k - 1.0) / 16.0
    q = (4.0 * k - 1.0) * (4.0 * k - 9.0) / 512.0
    c1 = -(4.0 * s1 - 3.0) / 16.0
    c2 = q[:, None, None] + q[None, :, None] + q[None, None, :]
    c2 = c2 + p[:, None, None] * p[None, :, None] + p[:, None, None] * p[None, None, :]
    c2 = c2 + p[None, :, None] * p[None, None, :]
    tail = 2.0 * t1 ** -0.5 + c1 * (2.0 / 3.0) * t1 ** -1.5 + c2 * 0.4 * t1 ** -2.5
    return g.reshape(n + 1, n + 1, n + 1) + (4.0 * math.pi) ** -1.5 * tail


def _convolve(fields):
    """G * f of real cubes (k, n, n, n)."""
    n = fields.shape[-1]
    g = _green(n - 1)
    i = torch.arange(2 * n, device="cuda")
    i = torch.where(i < n, i, 2 * n - i).clamp(max=n - 1)   # the entry at n meets zeros only
    kernel = -g[i][:, i][:, :, i]
    del g
    kh = torch.fft.rfftn(kernel)
    del kernel
    out = torch.empty_like(fields)
    for a in range(len(fields)):
        u = torch.fft.irfftn(torch.fft.rfftn(fields[a], s=(2 * n,) * 3) * kh, s=(2 * n,) * 3)
        out[a] = u[:n, :n, :n]
    return out


def _solve(blocks, n_b: int, fs):
    """The solution at the blocks' points for every source of the list."""
    nb = int(np.max(np.max(blocks, axis=0) - np.min(blocks, axis=0))) + 1
    side = nb * n_b
    b = torch.as_tensor(blocks - blocks.min(axis=0), device="cuda", dtype=torch.int64) * n_b
    r = torch.arange(n_b, device="cuda")
    at = ((b[:, 2, None, None, None] + r[None, :, None, None]) * side + b[:, 1, None, None, None]
          + r[None, None, :, None]) * side + b[:, 0, None, None, None] + r[None, None, None, :]
    at = at.reshape(-1)
    box = torch.zeros((len(fs), side ** 3), device="cuda", dtype=torch.float64)
    for i, f in enumerate(fs):
        box[i, at] = f.reshape(-1)
    u = _convolve(box.view(len(fs), side, side, side)).reshape(len(fs), -1)
    return [u[i, at].view(fs[i].shape) for i in range(len(fs))]


def exact(case, seed):
    # the sources as the solver gets them, rounded to its precision
    fs = [x.to(_PREC[case["prec"]][1]).double() for x in _sources(case, seed)]
    if case["kind"] == "conv":
        f = fs[0]
        n = case["n_b"]
        i = torch.arange(2 * n, device="cuda")
        i = torch.where(i < n, i, 2 * n - i).clamp(max=n - 1)
        kh = torch.fft.rfftn(-_green(n - 1)[i][:, i][:, :, i])
        step = max(1, (1 << 26) // (2 * n) ** 3)
        u = [torch.fft.irfftn(torch.fft.rfftn(f[a:a + step], s=(2 * n,) * 3, dim=(1, 2, 3)) * kh, s=(2 * n,) * 3,
                              dim=(1, 2, 3))[:, :n, :n, :n] for a in range(0, len(f), step)]
        return torch.cat(u)
    if case["kind"] == "batch":
        return [_solve(b, n_b, [f])[0] for (b, n_b, _, _), f in zip(_batch(case), fs)]
    u = _solve(_domain(case)[0], case["n_b"], fs)
    if case["kind"] == "multi":
        return torch.stack(u)
    return [x.cpu() for x in u] if case["kind"] == "host" else u[0]
