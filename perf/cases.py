"""The workloads that performance is measured on: what users of this library have it do.

A case fixes a surface (shape, size in metres, cells), the wavelength (1 m: k = 2 pi), the depth of the
oct-tree, the digits of the expansion, the arithmetic, the operation and the number of columns.  Meshes are the
repository's own families: icospheres whose edges are 0.07-0.15 wavelengths (cells = subdivisions), plates and cubes
of 0.1-wavelength squares split in two (cells = squares per side).  Right-hand sides are N(0, 1) columns, as Krylov
blocks and random probes are.

Operations (each one pass through the public binding):
  matvec    y = Z x
  adjoint   y = Z^H x
  x_r       X x (cos kernel) and R x (sin kernel), the two products of the characteristic-mode pencil
  gradient  y = Z(k) x through autograd, and the gradients of |y|^2 / 2 for x and for the wavenumber (dZ/dk)
  host      y = Z x between pinned host buffers
  sweep     y_f = Z(k_f) x_f at three wavenumbers (0.9, 1, 1.1 x nominal) through a plan set
"""
import functools
import math

import numpy as np
import torch

from paper_1412_1756_gb300 import mlfma

ETA = 376.730313668
K0 = float(np.float32(2.0 * math.pi))   # exactly representable in float32, so a float32 tensor can carry it
SWEEP = (0.9, 1.0, 1.1)
PRECISIONS = {"fp32": mlfma.FP32, "fp64": mlfma.FP64, "3xtf32": mlfma.MIXED_3XTF32}


def _case(name, shape, size, cells, levels, op, columns, prec="fp32", is_complex=False, digits=3.0):
    c = {"shape": shape, "size": size, "cells": cells, "levels": levels, "digits": digits, "prec": prec, "op": op,
         "columns": columns, "complex": is_complex}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one vector on the smallest sphere: what a call costs when launches and latency are all there is
        _case("sphere480-matvec-b1", "sphere", 1.0, 2, 3, "matvec", 1),
        # the small validation problem, all in FP64, eight columns
        _case("sphere1920-matvec-fp64-b8", "sphere", 1.0, 3, 3, "matvec", 8, prec="fp64"),
        # one complex Krylov vector: the product inside a single-vector iterative solve
        _case("sphere30720-matvec-complex1", "sphere", 4.0, 5, 5, "matvec", 1, is_complex=True),
        # the block eigensolver's product: 40 real columns
        _case("sphere30720-matvec-b40", "sphere", 4.0, 5, 5, "matvec", 40),
        # the pencil's two products for the ten modes nearest zero
        _case("sphere30720-x_r-b10", "sphere", 4.0, 5, 5, "x_r", 10),
        # an open flat surface with tensor-core interpolation
        _case("plate10680-matvec-3xtf32-b16", "plate", 6.0, 60, 5, "matvec", 16, prec="3xtf32"),
        # a differentiated product: value, gradient for the currents and for the wavenumber
        _case("plate10680-gradient-b8", "plate", 6.0, 60, 5, "gradient", 8),
        # a frequency sweep of a small closed body, an odd number of columns
        _case("cube7200-sweep-b7", "cube", 2.0, 20, 4, "sweep", 7),
        # the plain FP64 single-vector product: the refinement and residual products of the eigensolvers
        _case("cube28800-matvec-fp64-b1", "cube", 4.0, 40, 5, "matvec", 1, prec="fp64", digits=5.0),
        # the large cube, 64 columns in one pass (the benchmark's workload)
        _case("cube115200-matvec-b64", "cube", 8.0, 80, 6, "matvec", 64, digits=5.0),
        # a product between pinned host buffers, copies included
        _case("cube28800-host-b64", "cube", 4.0, 40, 5, "host", 64),
        # a large sphere with a ragged block of complex columns
        _case("sphere122880-adjoint-complex17", "sphere", 8.0, 6, 6, "adjoint", 17, is_complex=True),
    ]


def _unknowns(c):
    n = c["cells"]
    return {"sphere": 30 * 4 ** n, "plate": 3 * n * n - 2 * n, "cube": 18 * n * n}[c["shape"]]


def draw(rng):
    while True:
        op = rng.choices(["matvec", "adjoint", "x_r", "gradient", "host", "sweep"], [8, 4, 2, 3, 2, 2])[0]
        prec = rng.choices(["fp32", "fp64", "3xtf32"], [12, 3, 2])[0]
        if op not in ("matvec", "adjoint") and prec == "3xtf32":
            prec = "fp32"
        shape = rng.choice(["sphere", "plate", "cube"])
        if shape == "sphere":
            cells = rng.choices([2, 3, 4, 5, 6], [4, 4, 4, 3, 0.5])[0]
            size = round(2.0 ** (cells - 3) * rng.uniform(0.85, 1.1), 3)
            size = max(size, 0.85)
        else:
            cells = int(round(math.exp(rng.uniform(math.log(10), math.log(80)))))
            size = cells / 10.0
        levels = max(3, 1 + int(math.floor(math.log2(size / 0.25) + 1e-9)))   # leaf boxes of 0.25-0.5 wavelengths
        columns = int(round(math.exp(rng.uniform(0.0, math.log(64)))))
        if prec == "fp64":
            columns = min(columns, rng.randint(1, 8))
        is_complex = op in ("matvec", "adjoint", "host") and rng.random() < 0.3
        if is_complex:
            columns = max(1, columns // 2)
        c = _case(None, shape, size, cells, levels, op, columns, prec, is_complex)
        # at most the work of the large cube's 64 columns (an FP64 column costs about 20 FP32 ones)
        cost = _unknowns(c) * columns * (2 if is_complex else 1) * (20 if prec == "fp64" else 1)
        cost *= {"x_r": 2, "gradient": 6, "sweep": 3}.get(op, 1)
        if cost <= 115200 * 64 and _unknowns(c) * (3 if op == "sweep" else 1) <= 130000:
            return c


# ------------------------------------------------------------------ meshes ---
@functools.lru_cache(maxsize=32)
def _mesh(shape, size, cells):
    if shape == "sphere":
        return _icosphere(cells, size / 2)
    if shape == "plate":
        lat, tris = _square(cells)
        v = np.concatenate([lat * (size / cells) - size / 2, np.zeros((lat.shape[0], 1))], 1)
        return v, tris.astype(np.int32)
    return _cube(cells, size)


def _square(n):
    """Lattice points of n x n squares and the two triangles of each."""
    i, j = (a.reshape(-1) for a in np.meshgrid(np.arange(n), np.arange(n), indexing="ij"))
    p = i * (n + 1) + j
    q = p + n + 1
    tris = np.concatenate([np.stack([p, q, q + 1], 1), np.stack([p, q + 1, p + 1], 1)], 0)
    a, b = np.meshgrid(np.arange(n + 1), np.arange(n + 1), indexing="ij")
    return np.stack([a.reshape(-1), b.reshape(-1)], 1).astype(float), tris


def _cube(n, side):
    lat, tris = _square(n)
    pts, faces = [], []
    for axis in range(3):
        for high in (0, 1):
            u, v = ((axis + 1) % 3, (axis + 2) % 3) if high else ((axis + 2) % 3, (axis + 1) % 3)
            p = np.zeros((lat.shape[0], 3))
            p[:, axis] = n * high
            p[:, u], p[:, v] = lat[:, 0], lat[:, 1]
            faces.append(tris + len(pts) * lat.shape[0])
            pts.append(p)
    p = np.concatenate(pts).astype(np.int64)
    key, inv = np.unique((p[:, 0] * (n + 1) + p[:, 1]) * (n + 1) + p[:, 2], return_inverse=True)
    v = np.stack([key // (n + 1) ** 2, key // (n + 1) % (n + 1), key % (n + 1)], 1)
    return (v - n / 2.0) * (side / n), inv.reshape(-1)[np.concatenate(faces)].astype(np.int32)


def _icosphere(subdivisions, radius):
    g = (1.0 + math.sqrt(5.0)) / 2.0
    v = np.array([[s, t * g, 0] for s in (-1, 1) for t in (-1, 1)], float)
    v = np.concatenate([v, v[:, [2, 0, 1]], v[:, [1, 2, 0]]])
    d = np.linalg.norm(v[:, None] - v[None], axis=2)
    f = np.array([(a, b, c) for a in range(12) for b in range(a) for c in range(b)
                  if max(d[a, b], d[b, c], d[a, c]) < 2.1])
    out = np.einsum("ij,ij->i", np.cross(v[f[:, 1]] - v[f[:, 0]], v[f[:, 2]] - v[f[:, 0]]), v[f[:, 0]]) > 0
    f = np.where(out[:, None], f, f[:, [0, 2, 1]])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    for _ in range(subdivisions):
        e = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), axis=1)
        key, inv = np.unique(e[:, 0] * np.int64(v.shape[0]) + e[:, 1], return_inverse=True)
        m = v[key // v.shape[0]] + v[key % v.shape[0]]
        ab, bc, ca = inv.reshape(3, -1) + v.shape[0]
        v = np.concatenate([v, m / np.linalg.norm(m, axis=1, keepdims=True)])
        a, b, c = f.T
        f = np.concatenate([np.stack(t, 1) for t in ((a, ab, ca), (ab, b, bc), (ca, bc, c), (ab, bc, ca))])
    return v * radius, f.astype(np.int32)


# ------------------------------------------------------------ what is timed ---
def _inputs(case, seed):
    """Right-hand sides on the GPU, from the seed alone."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, b = _unknowns(case), case["columns"]
    shape = ((len(SWEEP), n, b) if case["op"] == "sweep" else (n, b)) + ((2,) if case["complex"] else ())
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64).to(torch.float64 if case["prec"] == "fp64" else torch.float32)
    return torch.view_as_complex(x) if case["complex"] else x


def _pinned(a):
    return torch.empty(a.shape, dtype=a.dtype, pin_memory=True).copy_(a).numpy()


def prepare(case, seed):
    v, t = _mesh(case["shape"], case["size"], case["cells"])
    cols = case["columns"] * (2 if case["complex"] else 1)
    prec = mlfma.FP64 if case["prec"] == "fp64" else mlfma.FP32
    s = {"op": case["op"], "prec": PRECISIONS[case["prec"]]}
    x = _inputs(case, seed)
    if case["op"] == "sweep":
        s["plan"] = mlfma.MlfmaPlanSet(v, t, [f * K0 for f in SWEEP], case["levels"], case["digits"], max_batch=cols, precisions=(prec,))
    else:
        s["plan"] = mlfma.MlfmaPlan(v, t, K0, case["levels"], case["digits"], max_batch=2 * cols if case["op"] == "gradient" else cols,
                                    precisions=(prec,))
    if case["op"] == "gradient":
        s["k"] = torch.tensor(K0, dtype=torch.float64 if prec == mlfma.FP64 else torch.float32, device="cuda", requires_grad=True)
        x.requires_grad_(True)
    if case["op"] == "host":
        s["x"] = _pinned(x)
        s["y"] = _pinned(torch.zeros(x.shape, dtype=torch.complex128 if prec == mlfma.FP64 else torch.complex64))
    else:
        s["x"] = x
    return s


def run(state):
    op, plan, x = state["op"], state["plan"], state["x"]
    if op == "matvec":
        return plan.matvec(x, prec=state["prec"])
    if op == "adjoint":
        return plan.matvec_adjoint(x, prec=state["prec"])
    if op == "x_r":
        return [plan.matvec_x(x), plan.matvec_r(x)]
    if op == "gradient":
        y = mlfma.efie_product(plan, x, state["k"])
        gx, gk = torch.autograd.grad(y, [x, state["k"]], y.detach())
        return {"y": y.detach(), "grad_x": gx, "grad_k": gk}
    if op == "host":
        return plan.matvec_host(x, prec=state["prec"], y=state["y"])
    return plan.matvec(x)


# ------------------------------------------------------------ what it costs ---
def _rwg(v, t):
    """One function per edge of two triangles, edges by (smaller, larger vertex): triangles (the one that runs along
    the edge from the smaller vertex first), local corners opposite the edge, lengths, midpoints."""
    t = t.astype(np.int64)
    a, b = t[:, [1, 2, 0]].reshape(-1), t[:, [2, 0, 1]].reshape(-1)   # the edge opposite corner 0, 1, 2
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    order = np.lexsort((a > b, hi, lo))
    key = (lo * np.int64(v.shape[0]) + hi)[order]
    two = np.flatnonzero(key[1:] == key[:-1])
    half = np.stack([order[two], order[two + 1]], 1)
    p, q = v[lo[half[:, 0]]], v[hi[half[:, 0]]]
    return half // 3, half % 3, np.linalg.norm(q - p, axis=1), (p + q) / 2


def _adjacent(key, weight, grid):
    """Sum of weight_m weight_m' over the pairs of occupied boxes that touch (each box with itself included)."""
    total = 0
    x, y, z = key // (grid * grid), key // grid % grid, key % grid
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                ok = (x + dx >= 0) & (x + dx < grid) & (y + dy >= 0) & (y + dy < grid) & (z + dz >= 0) & (z + dz < grid)
                k = key[ok] + (dx * grid + dy) * grid + dz
                at = np.minimum(np.searchsorted(key, k), key.size - 1)
                total += int((weight[ok] * weight[at] * (key[at] == k)).sum())
    return total


@functools.lru_cache(maxsize=64)
def _tree(shape, size, cells, levels, digits, k):
    """(N, near entries, per level 2.. (box count, translations, L))."""
    v, t = _mesh(shape, size, cells)
    mid = _rwg(v, t)[3]
    lo, hi = v.min(0), v.max(0)
    side = (hi - lo).max()
    corner = (lo + hi) / 2 - side / 2
    out, near = [], 0
    leaf = levels - 1
    ijk = np.clip(((mid - corner) / side * 2 ** leaf).astype(np.int64), 0, 2 ** leaf - 1)
    boxes = {}
    for l in range(leaf, 0, -1):
        g = 2 ** l
        c = ijk >> (leaf - l)
        key, count = np.unique((c[:, 0] * g + c[:, 1]) * g + c[:, 2], return_counts=True)
        boxes[l] = (key, count, g)
    near = _adjacent(*boxes[leaf])
    for l in range(2, levels):
        key, _, g = boxes[l]
        pk = (key // (g * g) // 2 * (g // 2) + key // g % g // 2) * (g // 2) + key % g // 2
        pkey, kids = np.unique(pk, return_counts=True)
        pairs = _adjacent(pkey, kids, g // 2) - _adjacent(key, np.ones(key.size, np.int64), g)
        kd = k * math.sqrt(3.0) * side / g
        out.append((key.size, pairs, math.ceil(kd + 1.8 * digits ** (2.0 / 3.0) * kd ** (1.0 / 3.0) - 1e-12)))
    return mid.shape[0], near, out


def _product_work(case, k, columns, rsize, taps=10):
    """One product Z x of `columns` real columns: x and y once, the near entries and leaf patterns once; the multiplications
    of the near field, the patterns, the translations, the separable interpolations and the shifts."""
    n, near, lv = _tree(case["shape"], case["size"], case["cells"], case["levels"], case["digits"], k)
    kl = 2 * (lv[-1][2] + 1) ** 2
    per = 4.0 * near + n * kl * 2 * (4 + 8)
    for i, (boxes, pairs, L) in enumerate(lv):
        K = 2 * (L + 1) ** 2
        per += pairs * K * 2 * 8
        if i + 1 < len(lv):
            kids, _, Lc = lv[i + 1]
            per += 2 * kids * 2 * ((L + 1) * 2 * (Lc + 1) * taps * 4 + K * taps * 4 + K * 8)
    return {"bytes": n * columns * 3 * rsize + (near + 2.0 * n * kl) * 2 * rsize, "flops": per * columns}


def work(case):
    r = 8 if case["prec"] == "fp64" else 4
    cols = case["columns"] * (2 if case["complex"] else 1)
    one = functools.partial(_product_work, case, rsize=r)
    if case["op"] == "x_r":
        parts = [one(K0, cols)] * 2
    elif case["op"] == "gradient":   # the value, the adjoint of a complex gradient, and dZ/dk (value and tangent)
        parts = [one(K0, cols), one(K0, 2 * cols), one(K0, 2 * cols)]
    elif case["op"] == "sweep":
        parts = [one(f * K0, cols) for f in SWEEP]
    else:
        parts = [one(K0, cols)]
    return {"bytes": float(sum(p["bytes"] for p in parts)), "flops": float(sum(p["flops"] for p in parts))}


# ------------------------------------------------- the same in 64 bits, dense ---
_S15 = math.sqrt(15.0)
_RULE = [(1 / 3, 1 / 3, 1 / 3, 9 / 40)]
for _c, _w in (((6 - _S15) / 21, (155 - _S15) / 1200), ((6 + _S15) / 21, (155 + _S15) / 1200)):
    _RULE += [(_c, _c, 1 - 2 * _c, _w), (_c, 1 - 2 * _c, _c, _w), (1 - 2 * _c, _c, _c, _w)]


class _Dense:
    """Products with the Galerkin matrix of the RWG functions, Z_ij = i k eta <f_i, (I - grad grad' / k^2) e^{ikR} / R, f_j>,
    and with dZ/dk, summed over all pairs of quadrature points (seven points a triangle) in 64 bits.  Triangle pairs whose
    centroids are closer than twice their longest edge take the 1/R part of the inner integral in closed form (the potentials
    of a uniform and a linear density on a flat triangle), averaged over both orders."""

    def __init__(self, v, t, device):
        f64 = dict(dtype=torch.float64, device=device)
        tri, corner, length, _ = _rwg(v, t)
        self.n, self.nt, self.dev = tri.shape[0], t.shape[0], device
        rule = torch.tensor(_RULE, **f64)
        self.w = rule[:, 3]
        self.p = torch.tensor(v[t], **f64)                                   # [nt, 3 corners, 3]
        nrm = torch.linalg.cross(self.p[:, 1] - self.p[:, 0], self.p[:, 2] - self.p[:, 0])
        self.area = 0.5 * torch.linalg.norm(nrm, dim=1)
        self.nrm = nrm / (2 * self.area)[:, None]
        self.q = torch.einsum("qc,tcd->tqd", rule[:, :3], self.p)            # [nt, 7, 3]
        sign = torch.tensor([1.0, -1.0], **f64)
        self.slot = torch.tensor((tri * 3 + corner).reshape(-1), device=device)   # half of a function -> (triangle, corner)
        self.half = (sign[None] * torch.tensor(length, **f64)[:, None]).reshape(-1) / (2 * self.area[self.slot // 3])
        self._near()

    def _near(self):
        cen, h = self.p.mean(1), (self.p - self.p[:, [1, 2, 0]]).norm(dim=2).amax(1)
        a = []
        for i in range(0, self.nt, 2048):
            d = (cen[i:i + 2048, None] - cen[None]).norm(dim=2)
            a.append((d < 2 * torch.maximum(h[i:i + 2048, None], h[None])).nonzero() + torch.tensor([i, 0], device=self.dev))
        self.a, self.b = torch.cat(a).T
        back = torch.argsort(self.b * self.nt + self.a)                      # the pair (b, a): the list is symmetric
        stat, phi = zip(*(self._static(self.a[i:i + 65536], self.b[i:i + 65536]) for i in range(0, self.a.numel(), 65536)))
        stat, phi = torch.cat(stat), torch.cat(phi)
        self.A0 = 0.5 * (stat + stat[back].transpose(1, 2))
        self.F0 = 0.5 * (phi + phi[back])

    def _static(self, a, b):
        """Blocks <f_a, 1/R, f_b> (corner functions r - p, 3 x 3) and <1, 1/R, 1>, the inner integral over b in closed form
        less the seven-point sum of 1/R that the sum over all points has (nothing at R = 0)."""
        r, n = self.q[a], self.nrm[b][:, None]
        h = ((r - self.p[b][:, :1]) * n).sum(2)
        rho = r - h[..., None] * n
        I0, I1 = torch.zeros_like(h), torch.zeros_like(r)
        for e in range(3):
            p0, p1 = self.p[b][:, e][:, None], self.p[b][:, (e + 1) % 3][:, None]
            length = (p1 - p0).norm(dim=2, keepdim=True)
            s = (p1 - p0) / length
            u = torch.linalg.cross(s, n.expand_as(s))
            lm, lp, d = ((p0 - rho) * s).sum(2), ((p1 - rho) * s).sum(2), ((p0 - rho) * u).sum(2)
            r0 = d * d + h * h
            rm, rp = torch.sqrt(r0 + lm * lm), torch.sqrt(r0 + lp * lp)
            on = r0 > 1e-26 * length[..., 0] ** 2
            safe = torch.where(on, r0, torch.ones_like(r0))
            f = torch.where(lm >= 0, torch.log((rp + lp) / torch.where(lm >= 0, rm + lm, rm).clamp_min(1e-300)),
                            torch.where(lp <= 0, torch.log((rm - lm) / torch.where(lp <= 0, rp - lp, rp).clamp_min(1e-300)),
                                        torch.log((rp + lp).clamp_min(1e-300) * (rm - lm).clamp_min(1e-300) / safe)))
            ah = h.abs()
            beta = torch.atan2(d * lp, r0 + ah * rp) - torch.atan2(d * lm, r0 + ah * rm)
            f, beta = torch.where(on, f, torch.zeros_like(f)), torch.where(on, beta, torch.zeros_like(f))
            I0 += d * f - ah * beta
            I1 += (0.5 * (r0 * f + lp * rp - lm * rm))[..., None] * u
        I1 += rho * I0[..., None]                                            # int r' / R
        R = (r[:, :, None] - self.q[b][:, None]).norm(dim=3)
        inv = torch.where(R > 0, 1 / R.clamp_min(1e-300), torch.zeros_like(R)) * (self.w * self.area[b][:, None])[:, None]
        I0 = I0 - inv.sum(2)
        I1 = I1 - torch.einsum("pqs,psd->pqd", inv, self.q[b])
        wo = self.w * self.area[a][:, None]
        ra = r[:, :, None] - self.p[a][:, None]                              # [pairs, 7, corner, 3]
        inner = I1[:, :, None] - self.p[b][:, None] * I0[..., None, None]
        return torch.einsum("pq,pqad,pqbd->pab", wo, ra, inner), (wo * I0).sum(1)

    def _spread(self, x):
        c = torch.zeros((self.nt * 3, x.shape[1]), dtype=x.dtype, device=self.dev)
        return c.index_add_(0, self.slot, self.half[:, None] * x.repeat_interleave(2, 0)).reshape(self.nt, 3, -1)

    def _gather(self, c):
        return (c.reshape(self.nt * 3, -1)[self.slot] * self.half[:, None]).reshape(self.n, 2, -1).sum(1)

    def products(self, x, ks, dk=False):
        """Z(k) x and, with dk, dZ/dk x for real columns x [N, B], at each k."""
        c = self._spread(x)
        nb = x.shape[1]
        wq = (self.w * self.area[:, None])
        rho = 2 * c.sum(1)
        J = torch.einsum("tqd,tb->tqdb", self.q, c.sum(1)) - torch.einsum("tcd,tcb->tdb", self.p, c)[:, None]
        src = (torch.cat([J, rho[:, None, None].expand(-1, 7, -1, -1)], 2) * wq[..., None, None]).reshape(self.nt * 7, 4 * nb)
        pts = self.q.reshape(-1, 3)
        out = []
        for k in ks:
            pot = torch.empty((2 if dk else 1, 2, pts.shape[0], 4 * nb), dtype=torch.float64, device=self.dev)
            step = max(1, int(2.5e8) // pts.shape[0])
            for i in range(0, pts.shape[0], step):
                R = torch.zeros((min(step, pts.shape[0] - i), pts.shape[0]), dtype=torch.float64, device=self.dev)
                for d in range(3):
                    R += (pts[i:i + step, d:d + 1] - pts[None, :, d]) ** 2
                R.sqrt_()
                s, co = torch.sin(k * R), torch.cos(k * R)
                if dk:                                                       # i e^{ikR}
                    pot[1, 0, i:i + step] = -(s @ src)
                    pot[1, 1, i:i + step] = co @ src
                own = R == 0
                R.masked_fill_(own, 1.0)
                pot[0, 0, i:i + step] = (co / R).masked_fill_(own, 0.0) @ src
                pot[0, 1, i:i + step] = (s / R).masked_fill_(own, k) @ src   # (e^{ikR} - 1) / R -> ik
            A, F = [], []
            for g in range(pot.shape[0]):
                pc = torch.complex(pot[g, 0], pot[g, 1]).reshape(self.nt, 7, 4, nb) * wq[..., None, None]
                va, ph = pc[:, :, :3], pc[:, :, 3]
                a = torch.einsum("tqd,tqdb->tb", self.q + 0j, va)[:, None] - torch.einsum("tcd,tdb->tcb", self.p + 0j, va.sum(1))
                f = 2 * ph.sum(1)
                if g == 0:
                    a = a.index_add_(0, self.a, torch.einsum("pab,pbc->pac", self.A0, c[self.b]) + 0j)
                    f = f.index_add_(0, self.a, 2 * self.F0[:, None] * rho[self.b] + 0j)
                A.append(self._gather(a))
                F.append(self._gather(f[:, None].expand(-1, 3, -1)))
            z = 1j * k * ETA * (A[0] - F[0] / k ** 2)
            out.append((z, 1j * ETA * (A[0] + F[0] / k ** 2) + 1j * k * ETA * (A[1] - F[1] / k ** 2)) if dk else z)
        return out

    def times(self, x, k):
        """Z x for real or complex x."""
        if not x.is_complex():
            return self.products(x.double(), [k])[0]
        z = self.products(torch.cat([x.real, x.imag], 1).double(), [k])[0]
        return z[:, :x.shape[1]] + 1j * z[:, x.shape[1]:]


def exact(case, seed):
    v, t = _mesh(case["shape"], case["size"], case["cells"])
    op = case["op"]
    cols = case["columns"] * (2 if case["complex"] else 1)
    cost = (7.0 * t.shape[0]) ** 2 * {"gradient": 5e-10 + 1e-10 * cols, "sweep": 3 * (3e-10 + 1.7e-11 * cols)}.get(op, 3e-10 + 1.7e-11 * cols)
    if cost > 14.0:
        return None
    x = _inputs(case, seed)
    D = _Dense(v, t, "cuda")
    if op == "x_r":
        z = D.times(x, K0)
        return [z.imag + 0j, z.real + 0j]
    if op == "adjoint":
        return D.times(x.conj().resolve_conj(), K0).conj().resolve_conj()
    if op == "gradient":
        y, dy = D.products(x.double(), [K0], dk=True)[0]
        return {"y": y, "grad_x": D.times(y.conj().resolve_conj(), K0).real, "grad_k": (y.conj() * dy).real.sum()}
    if op == "sweep":
        return torch.stack([D.times(x[i], f * K0) for i, f in enumerate(SWEEP)])
    y = D.times(x, K0)
    return y.cpu().numpy() if op == "host" else y
