"""Performance cases: the calls that a user of this library makes, over the sizes it is used at.

Four kinds of call, each through the public Python entry points:

  forward    ``api.spherical_harmonics``: values, with gradients or Hessians, in FP32,
             FP32 stored as bfloat16, FP64, or FP32 storage with FP64 arithmetic
  train      ``autograd.spherical_harmonics_autograd`` with its fused backward and, for
             force training, its double backward
  ragged     ``api.compute_batched``: many point sets, each with its own l_max
  expansion  ``api.expansion``: radial expansion of neighbour lists, per centre

``exact`` evaluates the same quantities in FP64 with plain torch: solid harmonics by their
three-term recursion in l, derivatives as linear maps from degree l - 1 to degree l.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2302_08381_gb300 import api
from paper_2302_08381_gb300.autograd import spherical_harmonics_autograd

DEV = "cuda"


def listed():
    return [
        # One MD step of a small structure: the edges of some 64 atoms, values and the
        # backward to positions. Launches and host latency count.
        dict(name="step_f32_l4_n2561", kind="train", n=2561, l_max=4, normalized=False, dtype="f32", second=False,
             points="shell"),
        # A reference-precision evaluation of a modest cloud, values only.
        dict(name="values_f64_l8_n10k", kind="forward", n=10_000, l_max=8, normalized=True, dtype="f64", order=0,
             points="normal"),
        # Values and gradients of a large edge list at a common l_max (the headline).
        dict(name="grad_f32_l8_n4M", kind="forward", n=4_194_304, l_max=8, normalized=False, dtype="f32", order=1,
             points="shell"),
        # The same for a mid-sized cloud at a higher l_max, stored as bfloat16 for a
        # 16-bit model downstream.
        dict(name="grad_bf16_l10_n1M", kind="forward", n=1_000_000, l_max=10, normalized=False, dtype="bf16",
             order=1, points="shell"),
        # Force training on a large batch of edges: forward, backward, and the backward of
        # the backward.
        dict(name="force_f32_l6_n4M", kind="train", n=4_194_304, l_max=6, normalized=False, dtype="f32", second=True,
             points="shell"),
        # High angular resolution (descriptors, wave-function work), many points at the poles.
        dict(name="grad_f32_l20_n200k", kind="forward", n=200_000, l_max=20, normalized=True, dtype="f32", order=1,
             points="poles"),
        # The highest degrees in common use.
        dict(name="grad_f32_l50_n200k", kind="forward", n=200_000, l_max=50, normalized=True, dtype="f32", order=1,
             points="poles"),
        # High degrees where FP64 accuracy is needed.
        dict(name="grad_f64_l30_n200k", kind="forward", n=200_000, l_max=30, normalized=True, dtype="f64", order=1,
             points="poles"),
        # Gradient-based fitting at high degree: forward and backward, an odd number of points.
        dict(name="step_f32_l30_n100k", kind="train", n=100_003, l_max=30, normalized=True, dtype="f32", second=False,
             points="shell"),
        # Serving many structures at once, each with its own l_max, into packed outputs.
        dict(name="ragged_512_sets", kind="ragged", nsets=512, nmin=1000, nmax=200_000, lset="3,6,8,12",
             normalized=False, size_seed=5),
        # Second derivatives (curvature, force constants).
        dict(name="hess_f32_l8_n400k", kind="forward", n=400_000, l_max=8, normalized=True, dtype="f32", order=2,
             points="shell"),
        # Density expansion coefficients of atomistic neighbour lists.
        dict(name="expansion_l6_c100k", kind="expansion", centres=100_000, mean=40, l_max=6, n_rad=8,
             normalized=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["forward"] * 6 + ["train"] * 3 + ["ragged", "expansion"])
    normalized = rng.random() < 0.5
    if kind == "forward":
        dtype = rng.choice(["f32", "f32", "f32", "bf16", "f64", "mixed"])
        order = rng.choice([0, 1, 1, 1, 2]) if dtype == "f32" else rng.choice([0, 1, 1])
        top = {"f32": 63, "bf16": 50, "f64": 50, "mixed": 50}[dtype] if order < 2 else 24
        l_max = _log_int(rng, 2, top + 1) - 1
        # as much output as the headline has, or as much FP64 arithmetic as the FP64 case
        planes = {0: 1, 1: 4, 2: 13}[order]
        cap = 1.3e9 / (planes * (l_max + 1) ** 2)
        if dtype in ("f64", "mixed"):
            cap = min(cap, 1.9e8 / (l_max + 1) ** 2)
        n = _log_int(rng, 1000, max(2000, min(4_000_000, int(cap))))
        # r^l stays well inside FP32 for the scaled form
        points = "poles" if l_max > 16 else rng.choice(["shell", "normal"])
        return dict(kind=kind, n=n, l_max=l_max, normalized=normalized, dtype=dtype, order=order, points=points)
    if kind == "train":
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        second = rng.random() < 0.3
        l_max = _log_int(rng, 2, 12 if second or dtype == "f64" else 64) - 1
        cap = min(4_000_000, int((1e7 if dtype == "f64" else 2e8) / (l_max + 1) ** 2))
        n = _log_int(rng, 500, max(1000, cap))
        points = "poles" if l_max > 16 else rng.choice(["shell", "normal"])
        return dict(kind=kind, n=n, l_max=l_max, normalized=normalized, dtype=dtype, second=second, points=points)
    if kind == "ragged":
        lset = ",".join(str(l) for l in sorted(rng.sample(range(1, 17), rng.randint(1, 5))))
        return dict(kind=kind, nsets=_log_int(rng, 4, 512), nmin=rng.choice([17, 200, 1000]),
                    nmax=_log_int(rng, 2000, 30_000), lset=lset, normalized=normalized,
                    size_seed=rng.randrange(1 << 20))
    return dict(kind=kind, centres=_log_int(rng, 100, 100_000), mean=rng.randint(4, 40), l_max=rng.randint(1, 8),
                n_rad=rng.randint(1, 8), normalized=normalized)


# ------------------------------------------------------------------ inputs


def _points(n, how, gen, dtype):
    d = torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64)
    if how == "normal":
        return d.to(dtype)
    d /= d.norm(dim=1, keepdim=True).clamp_min(1e-300)
    if how == "shell":
        return (d * (0.7 + 4.3 * torch.rand(n, 1, generator=gen, device=DEV, dtype=torch.float64))).to(dtype)
    # half of them on the unit sphere, half within 1e-4 rad of the poles
    th = 1e-4 * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    ph = 2 * math.pi * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    sg = 1.0 - 2.0 * (torch.arange(n, device=DEV) % 4 >= 2).double()
    pole = torch.stack([th.sin() * ph.cos(), th.sin() * ph.sin(), sg * th.cos()], 1)
    return torch.where((torch.arange(n, device=DEV) % 2 == 0)[:, None], d, pole).to(dtype)


def _sets(case):
    """Sizes and l_max of a ragged batch, and where each set's outputs start."""
    rng = np.random.default_rng(case["size_seed"])
    sizes = np.rint(np.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["nsets"]))).astype(int)
    ls = rng.choice([int(l) for l in case["lset"].split(",")], case["nsets"])
    out, at = [], 0
    for n, l in zip(sizes.tolist(), ls.tolist()):
        out.append((n, l, at))
        at += -(-n * (l + 1) ** 2 // 64) * 64  # every set starts on a 256-byte boundary
    return out, at


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    st = dict(case)
    if case["kind"] == "ragged":
        sets, total = _sets(case)
        st["xyz"] = [torch.randn(n, 3, generator=gen, device=DEV) for n, _, _ in sets]
        st["ls"] = [l for _, l, _ in sets]
        st["sph"] = torch.zeros(total, device=DEV)
        st["dsph"] = torch.zeros(3 * total, device=DEV)
        st["outputs"] = []
        for n, l, at in sets:
            K = (l + 1) ** 2
            st["outputs"].append((st["sph"][at:at + n * K].view(n, K),
                                  st["dsph"][3 * at:3 * (at + n * K)].view(n, 3, K)))
        return st
    if case["kind"] == "expansion":
        counts = torch.randn(case["centres"], generator=gen, device=DEV) * (case["mean"] / 4) + case["mean"]
        counts = counts.round().clamp(0, 3 * case["mean"]).long()
        st["offsets"] = torch.cat([torch.zeros(1, dtype=torch.long, device=DEV), counts.cumsum(0)])
        edges = int(st["offsets"][-1])
        st["xyz"] = _points(edges, "shell", gen, torch.float32)
        st["radial"] = torch.randn(edges, case["n_rad"], case["l_max"] + 1, generator=gen, device=DEV)
        return st
    dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
    st["xyz"] = _points(case["n"], case["points"], gen, dtype)
    if case["kind"] == "train":
        K = (case["l_max"] + 1) ** 2
        st["xyz"].requires_grad_(True)
        st["g"] = torch.randn(case["n"], K, generator=gen, device=DEV, dtype=dtype).requires_grad_(case["second"])
        st["v"] = torch.randn(case["n"], 3, generator=gen, device=DEV, dtype=dtype)
    return st


# --------------------------------------------------------------------- run


def run(st):
    kind = st["kind"]
    if kind == "forward":
        return api.spherical_harmonics(
            st["xyz"], st["l_max"], normalized=st["normalized"], gradients=st["order"] >= 1,
            hessians=st["order"] == 2, out_dtype=torch.bfloat16 if st["dtype"] == "bf16" else None,
            qprec="f64" if st["dtype"] == "mixed" else "native")
    if kind == "train":
        x, g = st["xyz"], st["g"]
        y = spherical_harmonics_autograd(x, st["l_max"], st["normalized"])
        (gx,) = torch.autograd.grad(y, x, g, create_graph=st["second"])
        if not st["second"]:
            return y, gx
        gg, gxx = torch.autograd.grad(gx, (g, x), st["v"])
        return y, gx, gg, gxx
    if kind == "ragged":
        api.compute_batched(st["xyz"], st["ls"], normalized=st["normalized"], outputs=st["outputs"])
        return st["sph"], st["dsph"]
    return api.expansion(st["xyz"], st["radial"], st["offsets"], st["l_max"], normalized=st["normalized"])


# -------------------------------------------------------------------- work


def work(case):
    # about 4 operations of the recursion per pair of columns (l, +-m), and 2 per output
    if case["kind"] == "ragged":
        b = f = 0
        for n, l, _ in _sets(case)[0]:
            K = (l + 1) ** 2
            b += n * (12 + 16 * K)
            f += n * 10 * K
        return {"bytes": b, "flops": f}
    K = (case["l_max"] + 1) ** 2
    if case["kind"] == "expansion":
        e, R = case["centres"] * case["mean"], case["n_rad"]
        return {"bytes": e * (12 + 4 * R * (case["l_max"] + 1)) + case["centres"] * (8 + 4 * R * K),
                "flops": e * K * (4 + 2 * R)}
    size = {"f32": 4, "bf16": 2, "f64": 8, "mixed": 4}[case["dtype"]]
    if case["kind"] == "forward":
        planes = {0: 1, 1: 4, 2: 13}[case["order"]]
        return {"bytes": case["n"] * (3 * (8 if case["dtype"] == "f64" else 4) + size * planes * K),
                "flops": case["n"] * K * (2 + 2 * planes)}
    # forward: xyz -> y; backward: xyz, g -> gx; double backward: xyz, g, v -> gg, gxx
    b = 3 + K + 3 + K + 3 + (9 + 2 * K + 3 if case["second"] else 0)
    return {"bytes": case["n"] * size * b, "flops": case["n"] * K * (12 + (20 if case["second"] else 0))}


# ------------------------------------------------------------------- exact


_MAPS = {}


def _maps(l):
    """The matrices of d/dx, d/dy, d/dz from the solid harmonics of degree l - 1 to those of degree l."""
    if l in _MAPS:
        return _MAPS[l]
    M = np.zeros((3, 2 * l + 1, max(2 * l - 1, 1)))
    r = math.sqrt((2 * l + 1) / (2 * l - 1)) if l else 0.0

    def put(i, m, mm, c):  # the coefficient of component mm of degree l - 1 in component m of degree l
        if abs(mm) <= l - 1:
            M[i, l + m, l - 1 + mm] += c

    for m in range(0, l + 1) if l else ():
        a = 0.5 * r * math.sqrt((l + m) * (l + m - 1))
        b = 0.5 * r * math.sqrt((l - m) * max(l - m - 1, 0))
        c = r * math.sqrt((l - m) * (l + m))
        if m == 0:
            put(0, 0, 1, -math.sqrt(2) * b)
            put(1, 0, -1, -math.sqrt(2) * b)
            put(2, 0, 0, c)
            continue
        w = math.sqrt(2) if m == 1 else 1.0  # the component m = 0 carries a factor 1/sqrt(2)
        put(0, m, m - 1, a * w)
        put(0, m, m + 1, -b)
        put(0, -m, -(m + 1), -b)
        put(1, m, -(m + 1), -b)
        put(1, -m, m - 1, a * w)
        put(1, -m, m + 1, b)
        if m > 1:
            put(0, -m, -(m - 1), a)
            put(1, m, -(m - 1), -a)
        put(2, m, m, c)
        put(2, -m, -m, c)
    _MAPS[l] = [torch.from_numpy(M[i]).to(DEV) for i in range(3)]
    return _MAPS[l]


def _solid(p, l_max):
    """[2l+1, n] solid harmonics of every degree l <= l_max at p [n, 3], FP64."""
    x, y, z = p.T
    r2 = (p * p).sum(1)
    Y = [torch.full((1, p.shape[0]), 1 / math.sqrt(4 * math.pi), dtype=torch.float64, device=p.device)]
    for l in range(1, l_max + 1):
        B = torch.empty(2 * l + 1, p.shape[0], dtype=torch.float64, device=p.device)
        m = torch.arange(-(l - 1), l, dtype=torch.float64, device=p.device)
        A = torch.sqrt((4 * l * l - 1) / (l * l - m * m))
        B[1:-1] = A[:, None] * z * Y[l - 1]
        if l >= 2:
            q = torch.sqrt((2 * l + 1) / (2 * l - 3) * ((l - 1) ** 2 - m * m) / (l * l - m * m))
            B[2:-2] -= q[1:-1, None] * r2 * Y[l - 2]
        s = math.sqrt((2 * l + 1) / (2 * l))
        c0 = Y[l - 1][-1] * (math.sqrt(2) if l == 1 else 1.0)
        s0 = Y[l - 1][0] if l > 1 else torch.zeros_like(x)
        B[-1] = s * (x * c0 - y * s0)
        B[0] = s * (x * s0 + y * c0)
        Y.append(B)
    return Y


def _reference(p, l_max, normalized, order):
    """Values [n, K], gradients [n, 3, K] and Hessians [n, 3, 3, K] at p (FP64), up to `order`."""
    n, K = p.shape[0], (l_max + 1) ** 2
    r = p.norm(dim=1)
    u = p / r[:, None] if normalized else p
    Y = _solid(u, l_max)
    out = [torch.cat(Y).T]
    if order >= 1:
        D = torch.zeros(n, 3, K, dtype=torch.float64, device=p.device)
        G = {}
        for l in range(1, l_max + 1):
            for i in range(3):
                G[l, i] = _maps(l)[i] @ Y[l - 1]
                g = (G[l, i] - l * u[:, i] * Y[l]) / r if normalized else G[l, i]
                D[:, i, l * l:(l + 1) ** 2] = g.T
        out.append(D)
    if order >= 2:
        H = torch.zeros(n, 3, 3, K, dtype=torch.float64, device=p.device)
        for l in range(1, l_max + 1):
            for i in range(3):
                for j in range(3):
                    h = (_maps(l)[i] @ _maps(l - 1)[j]) @ Y[l - 2] if l >= 2 else torch.zeros_like(Y[l])
                    if normalized:
                        h = h - l * (u[:, i] * G[l, j] + u[:, j] * G[l, i]) + l * (l + 2) * u[:, i] * u[:, j] * Y[l]
                        h = (h - l * Y[l] if i == j else h) / r**2
                    H[:, i, j, l * l:(l + 1) ** 2] = h.T
        out.append(H)
    return out


def _chunks(n, l_max, order):
    step = max(1024, int(2e8 // ((l_max + 1) ** 2 * {0: 2, 1: 8, 2: 26}[order])))
    return [slice(a, min(a + step, n)) for a in range(0, n, step)]


def exact(case, seed):
    st = prepare(case, seed)
    if case["kind"] == "forward":
        p, l = st["xyz"].double(), case["l_max"]
        K, n, order = (l + 1) ** 2, case["n"], case["order"]
        outs = [torch.empty(n, *lead, K, dtype=torch.float64, device=DEV) for lead in [(), (3,), (3, 3)][:order + 1]]
        for c in _chunks(n, l, order):
            for o, v in zip(outs, _reference(p[c], l, case["normalized"], order)):
                o[c] = v
        return outs[0] if order == 0 else tuple(outs)
    if case["kind"] == "train":
        p, g, v = st["xyz"].detach().double(), st["g"].detach().double(), st["v"].double()
        order = 2 if case["second"] else 1
        parts = []
        for c in _chunks(case["n"], case["l_max"], order):
            R = _reference(p[c], case["l_max"], case["normalized"], order)
            t = [R[0], torch.einsum("nik,nk->ni", R[1], g[c])]
            if case["second"]:
                t += [torch.einsum("nik,ni->nk", R[1], v[c]), torch.einsum("nijk,nk,nj->ni", R[2], g[c], v[c])]
            parts.append(t)
        return tuple(torch.cat(t) for t in zip(*parts))
    if case["kind"] == "ragged":
        sets, total = _sets(case)
        sph = torch.zeros(total, dtype=torch.float64, device=DEV)
        dsph = torch.zeros(3 * total, dtype=torch.float64, device=DEV)
        for (n, l, at), x in zip(sets, st["xyz"]):
            K = (l + 1) ** 2
            y, d = _reference(x.double(), l, case["normalized"], 1)
            sph[at:at + n * K] = y.reshape(-1)
            dsph[3 * at:3 * (at + n * K)] = d.reshape(-1)
        return sph, dsph
    l, off = case["l_max"], st["offsets"]
    K = (l + 1) ** 2
    of = torch.repeat_interleave(torch.arange(case["centres"], device=DEV), off[1:] - off[:-1])
    lv = torch.tensor([a for a in range(l + 1) for _ in range(2 * a + 1)], device=DEV)
    out = torch.zeros(case["centres"], case["n_rad"], K, dtype=torch.float64, device=DEV)
    for c in _chunks(st["xyz"].shape[0], l, 2):
        (y,) = _reference(st["xyz"][c].double(), l, case["normalized"], 0)
        out.index_add_(0, of[c], st["radial"][c].double()[:, :, lv] * y[:, None, :])
    return out
