"""The work that users of this library have it do, as cases that can be timed.

Every case is one pass through the public entry points (`Plan`, `Batch`,
`Upward`, `triangles_single`) on seeded synthetic meshes in octree leaves.
`listed()` are fixed cases, `draw(rng)` gives others from the same ranges,
`prepare` makes what a program holds before the call, `run` is the call,
`work` what it cannot do without, and `exact` the outputs from plain torch in
64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2107_10942_gb300 as q2x
from paper_2107_10942_gb300.q2x import Batch, triangles_single
from paper_2107_10942_gb300.upward import Upward

DEV = "cuda"
NV = {"segment": 2, "triangle": 3, "tetra": 4}
DIM = {"segment": 1, "triangle": 2, "tetra": 3}


# --------------------------------------------------------------------- cases


def listed():
    return [
        # A small closed surface as one expansion: the shortest call, bound by
        # latency and launches (level-3 icosphere size, 1,280 triangles).
        _elements("one-leaf-fp64", "triangle", 8, 0, 10, "fp64"),
        # The precision workload: a large surface mesh (5,242,880 triangles)
        # in 60 thousand leaves, FP64 ...
        _elements("sphere-large-fp64", "triangle", 512, 7, 16, "fp64"),
        # ... and the same call in the FP32-mixed mode.
        _elements("sphere-large-fp32", "triangle", 512, 7, 16, "fp32"),
        # A boundary-element surface with vertex densities, single and double
        # layer in one pass (327,680 triangles), FP64.
        _elements("sphere-linear-both-fp64", "triangle", 128, 5, 12, "fp64", density="linear", double=True),
        # Filaments, surface and volume elements in one adaptive octree with a
        # degree per leaf, replayed as one batch (FP32-mixed).
        dict(name="mixed-batch-fp32", op="batch", n_fil=2000, n_steps=1000, freq=447, grid=64, max_leaf=2000, p_lo=8,
             p_hi=20, precision="fp32"),
        # Shape optimisation: forward and gradient (vertices, densities) of the
        # single layer on a million triangles, FP32-mixed.
        dict(name="adjoint-fp32", op="adjoint", freq=224, depth=6, p=12, precision="fp32"),
        # Line currents: vector coefficients of two million filament segments,
        # and the Biot-Savart field of a root expansion at 2^18 targets.
        dict(name="line-currents-fp64", op="currents", n_fil=2000, n_steps=1000, depth=6, p=12, n_tgt=262144),
        # The upward pass of an octree over a surface's leaves.
        dict(name="upward-fp64", op="upward", freq=128, depth=5, p=12),
        # Far field of a few expansions at many targets.
        dict(name="far-field-fp64", op="far", n_exp=1, per_target=1, n_tgt=1048576, p=12, norm="coeff"),
        # Exact near field: collocation of a surface's triangles, each against
        # the triangles of its leaf (the self term among them).
        dict(name="near-field-fp64", op="near", kind="triangle", freq=128, depth=5, layer=0),
        # Receiver side of a Galerkin method: local expansions integrated over
        # the surface's triangles.
        dict(name="galerkin-fp64", op="galerkin", freq=128, depth=5, p=12, layer=0),
        # Per-element rows that a program made itself, summed into leaves.
        dict(name="leaf-reduce-fp64", op="reduce", freq=128, depth=5, p=12),
    ]


def _elements(name, kind, size, depth, p, precision, density="const", single=True, double=False, norm="coeff",
              rho=True, ragged=False):
    c = dict(op="elements", kind=kind, size=size, depth=depth, p=p, precision=precision, density=density,
             single=single, double=double, norm=norm, rho=rho, ragged=ragged)
    if name:
        c["name"] = name
    return c


def _count(kind, size):
    return {"triangle": 20 * size * size, "segment": size * size, "tetra": 6 * size ** 3}[kind]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _depth_for(rng, n, surface=True):
    """An octree depth that leaves about 8 to 200 elements in a leaf (0: one leaf)."""
    if n < 400 and rng.random() < 0.5:
        return 0
    per = math.exp(rng.uniform(math.log(8), math.log(200)))
    boxes = max(1.0, n / per)
    d = math.log(max(1.0, boxes / 4), 4) if surface else math.log(boxes, 8)
    return max(0, min(8, int(round(d))))


def draw(rng):
    op = rng.choice(["elements"] * 5 + ["batch", "adjoint", "currents", "upward", "far", "near", "galerkin", "reduce"])
    p = rng.randint(2, 20)
    if op == "elements":
        kind = rng.choice(["triangle", "triangle", "triangle", "segment", "tetra"])
        precision = rng.choice(["fp64", "fp64", "fp32"])
        density = rng.choice(["const", "linear"]) if kind == "triangle" else "const"
        layers = rng.choice([(True, False), (True, True), (False, True)]) if kind == "triangle" else (True, False)
        levels = {"segment": 2, "triangle": 3, "tetra": 4}[kind] + (2 if density == "linear" else 0) + layers[1]
        most = 5242880 * 289 * 3 / ((p + 1) ** 2 * levels)  # elements: no more work than the largest listed case
        most = min(most, 5242880)
        lo, hi = {"triangle": (2, math.sqrt(most / 20)), "segment": (6, math.sqrt(most)),
                  "tetra": (2, (most / 6) ** (1 / 3))}[kind]
        size = _log_int(rng, lo, hi)
        n = _count(kind, size)
        return _elements(None, kind, size, _depth_for(rng, n, kind != "tetra"), p, precision, density, *layers,
                         norm=rng.choice(["coeff", "coeff", "moment"]), rho=rng.random() < 0.8,
                         ragged=rng.random() < 0.25)
    if op == "batch":
        return dict(op=op, n_fil=_log_int(rng, 4, 1500), n_steps=_log_int(rng, 30, 900), freq=_log_int(rng, 10, 400),
                    grid=_log_int(rng, 4, 56), max_leaf=_log_int(rng, 200, 3000), p_lo=min(p, 8), p_hi=max(p, 8),
                    precision=rng.choice(["fp32", "fp32", "fp64"]) if p <= 12 else "fp32")
    f = _log_int(rng, 5, 200)
    d = max(1, _depth_for(rng, 20 * f * f))
    if op == "adjoint":
        return dict(op=op, freq=f, depth=d, p=min(p, 16), precision=rng.choice(["fp32", "fp64"]) if f < 60 else "fp32")
    if op == "currents":
        nf, ns = _log_int(rng, 3, 1500), _log_int(rng, 20, 900)
        return dict(op=op, n_fil=nf, n_steps=ns, depth=_depth_for(rng, nf * ns, False), p=min(p, 16),
                    n_tgt=_log_int(rng, 100, 200000))
    if op == "upward":
        return dict(op=op, freq=f, depth=min(max(d, 2), 6), p=min(p, 16))
    if op == "far":
        k = rng.choice([1, 1, 2, 5, 8])
        return dict(op=op, n_exp=rng.choice([k, k + 7, 64 + k, 500]), per_target=k,
                    n_tgt=_log_int(rng, 100, 1000000 // k), p=min(p, 16), norm=rng.choice(["coeff", "coeff", "moment"]))
    if op == "near":
        kind = rng.choice(["triangle", "triangle", "segment"])
        f = _log_int(rng, 4, 90)
        return dict(op=op, kind=kind, freq=f, depth=max(0, _depth_for(rng, 20 * f * f)),
                    layer=rng.choice([0, 1]) if kind == "triangle" else 0)
    if op == "galerkin":
        return dict(op=op, freq=f, depth=d, p=min(p, 16), layer=rng.choice([0, 1]))
    return dict(op="reduce", freq=min(f, 150), depth=d, p=min(p, 14))


# ------------------------------------------------------------------- geometry


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape, lo=-1.0, hi=1.0):
    return torch.rand(*shape, dtype=torch.float64, device=DEV, generator=g) * (hi - lo) + lo


def _sphere(freq, g):
    """A geodesic sphere (20 freq^2 triangles) with a smooth random bump of a tenth of its radius."""
    t = (1.0 + math.sqrt(5.0)) / 2.0
    v = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                  [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]], dtype=np.float64)
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    f = np.array([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                  [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5],
                  [2, 4, 11], [6, 2, 10], [8, 6, 7], [9, 8, 1]])
    corner = torch.from_numpy(v[f]).to(DEV)  # (20, 3, 3)
    i, j = torch.meshgrid(torch.arange(freq + 1, device=DEV), torch.arange(freq + 1, device=DEV), indexing="ij")
    keep = (i + j <= freq)
    num = torch.full((freq + 1, freq + 1), -1, dtype=torch.int64, device=DEV)
    nl = (freq + 1) * (freq + 2) // 2
    num[keep] = torch.arange(nl, device=DEV)
    b = torch.stack([freq - i[keep] - j[keep], i[keep], j[keep]]).double() / freq  # barycentric (3, nl)
    y = torch.einsum("kl,fkd->dfl", b, corner).reshape(3, -1)
    y = y / y.norm(dim=0, keepdim=True)
    up = torch.stack([num[:-1, :-1], num[1:, :-1], num[:-1, 1:]])[:, (i + j < freq)[:-1, :-1]]
    dn = torch.stack([num[1:, :-1], num[1:, 1:], num[:-1, 1:]])[:, (i + j < freq - 1)[:-1, :-1]]
    tri = torch.cat([up, dn], dim=1)
    tri = (tri[:, None, :] + (torch.arange(20, device=DEV) * nl)[None, :, None]).reshape(3, -1)
    wave = 3.0 * torch.randn(8, 3, dtype=torch.float64, device=DEV, generator=g)
    bump = torch.cos(wave @ y + _uniform(g, 8, 1, hi=math.pi)).sum(0)
    return y * (1.0 + 0.1 * bump / bump.abs().max()), tri


def _filaments(n_fil, n_steps, g):
    """Random walks of steps 1e-3 in the unit ball; two vertices a segment, shared along a filament."""
    start = torch.randn(3, n_fil, dtype=torch.float64, device=DEV, generator=g)
    start = start / start.norm(dim=0) * 0.9 * _uniform(g, n_fil, lo=0.0) ** (1 / 3)
    step = torch.randn(3, n_fil, n_steps, dtype=torch.float64, device=DEV, generator=g)
    step = 1e-3 * step / step.norm(dim=0)
    walk = torch.cat([start[:, :, None], start[:, :, None] + step.cumsum(2)], dim=2)
    a = torch.arange(n_fil, device=DEV)[:, None] * (n_steps + 1) + torch.arange(n_steps, device=DEV)[None]
    return walk.reshape(3, -1), torch.stack([a, a + 1]).reshape(2, -1)


def _tets(grid, g):
    """Six tetrahedra a cell of a jittered grid in the unit ball's cube."""
    n, h = grid + 1, 1.0 / grid
    ax = torch.arange(n, device=DEV)
    i, j, k = torch.meshgrid(ax, ax, ax, indexing="ij")
    v = torch.stack([i, j, k]).reshape(3, -1).double() * (1.15 * h) - 0.575
    v = v + _uniform(g, 3, v.shape[1], lo=-0.15 * h, hi=0.15 * h)
    cell = ((i * n + j) * n + k)[:-1, :-1, :-1].reshape(-1)
    step = {0: n * n, 1: n, 2: 1}
    out = []
    for a, b, c in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        o1, o2 = step[a], step[a] + step[b]
        out.append(torch.stack([cell, cell + o1, cell + o2, cell + o2 + step[c]]))
    return v, torch.cat(out, dim=1)


def _morton(ijk, depth):
    code = torch.zeros_like(ijk[0])
    for b in range(depth):
        for d in range(3):
            code |= ((ijk[d] >> b) & 1) << (3 * b + 2 - d)
    return code


def _unmorton(code, depth):
    ijk = [torch.zeros_like(code) for _ in range(3)]
    for b in range(depth):
        for d in range(3):
            ijk[d] |= ((code >> (3 * b + 2 - d)) & 1) << b
    return torch.stack(ijk)


def _cells(v, el, lo, size, depth):
    c = v[:, el].mean(1)
    ijk = ((c - lo) / size * (1 << depth)).floor().to(torch.int64).clamp_(0, (1 << depth) - 1)
    return _morton(ijk, depth)


def _leaf_rho(v, el, leaf, leaf_c, out=None):
    out = torch.zeros(leaf_c.shape[1], dtype=torch.float64, device=DEV) if out is None else out
    for k in range(el.shape[0]):
        out.scatter_reduce_(0, leaf, (v[:, el[k]] - leaf_c[:, leaf]).norm(dim=0), "amax")
    return out


def _moved(v, g, amp):
    """The mesh of this seed: the leaves belong to the case's mesh, the vertices move a little within them."""
    return (v + amp * _uniform(g, *v.shape)).contiguous()


def _in_leaves(v, el, lo, size, depth, g, amp):
    """Elements sorted into the non-empty leaves of a uniform octree."""
    code, order = torch.sort(_cells(v, el, lo, size, depth), stable=True)
    el = el[:, order]
    uniq, leaf, counts = torch.unique_consecutive(code, return_inverse=True, return_counts=True)
    off = torch.zeros(uniq.numel() + 1, dtype=torch.int64, device=DEV)
    off[1:] = counts.cumsum(0)
    c = lo + (_unmorton(uniq, depth).double() + 0.5) * (size / (1 << depth))
    v = _moved(v, g, amp)
    return dict(vxyz=v, idx=el.to(torch.int32).contiguous(), el=el, leaf=leaf, leaf_off=off,
                leaf_c=c.contiguous(), leaf_rho=_leaf_rho(v, el, leaf, c))


def _mesh(kind, size, g):
    """Vertices, elements, the octree's corner and width, and how far vertices may move."""
    if kind == "triangle":
        return _sphere(size, g) + (-1.125, 2.25, 0.1 / size)
    if kind == "segment":
        return _filaments(size, size, g) + (-1.25, 2.5, 1e-4)
    return _tets(size, g) + (-0.75, 1.5, 0.05 / size)


def _inputs(c, seed):
    """The inputs of a case (geometry, densities, weights), from the seed alone."""
    g, op = _gen(seed), c["op"]
    mesh = _gen(20210710)  # one mesh and one set of leaves a case, moved and loaded by the seed
    if op == "batch":
        return _batch_inputs(c, g, mesh)
    if op in ("currents", "far"):
        s = {}
        if op == "currents":
            v, el = _filaments(c["n_fil"], c["n_steps"], mesh)
            s = _in_leaves(v, el, -1.25, 2.5, c["depth"], g, 1e-4)
            t = s["vxyz"][:, s["el"][1]] - s["vxyz"][:, s["el"][0]]
            s["current"] = (t / t.norm(dim=0) * _uniform(g, t.shape[1])).contiguous()
        n_exp = 1 if op == "currents" else c["n_exp"]
        comp = 3 if op == "currents" else 1
        s["exp_c"] = _uniform(g, 3, n_exp, lo=-0.5, hi=0.5) if op == "far" else torch.zeros(3, 1, dtype=torch.float64, device=DEV)
        rho = _uniform(g, n_exp, lo=0.2, hi=0.8)
        s["coef"] = torch.stack([_rows(g, n_exp, c["p"], rho, c.get("norm", "coeff")) for _ in range(comp)])
        x = torch.randn(3, c["n_tgt"], dtype=torch.float64, device=DEV, generator=g)
        s["tgt"] = (x / x.norm(dim=0) * _uniform(g, c["n_tgt"], lo=2.0, hi=3.0)).contiguous()
        k = c.get("per_target", 1)
        s["tgt_off"] = torch.arange(c["n_tgt"] + 1, dtype=torch.int64, device=DEV) * k
        first = torch.randint(0, n_exp, (c["n_tgt"], 1), device=DEV, generator=g)
        s["exp_idx"] = ((first + torch.arange(k, device=DEV)) % n_exp).reshape(-1).contiguous()
        return s
    kind = c.get("kind", "triangle")
    size = c["size"] if op == "elements" else c["freq"]
    if op == "near" and kind == "segment":
        size = int(math.sqrt(20) * size)
    v, el, lo, width, amp = _mesh(kind, size, mesh)
    s = _in_leaves(v, el, lo, width, c["depth"], g, amp)
    s.update(lo=lo, width=width)
    n, n_leaves = el.shape[1], s["leaf_c"].shape[1]
    s["sigma"] = _uniform(g, v.shape[1] if c.get("density") == "linear" else n)
    s["leaf_p"] = None
    if c.get("ragged"):
        s["leaf_p"] = torch.randint(c["p"] // 2, c["p"] + 1, (n_leaves,), device=DEV, generator=g).to(torch.int32)
    if op == "near":
        s["tgt"] = s["vxyz"][:, s["el"]].mean(1)
        if c["layer"] or kind == "segment":  # off the elements themselves
            s["tgt"] = s["tgt"] * (1.0 + 0.2 / size)
        s["tgt"] = s["tgt"].contiguous()
        per = torch.diff(s["leaf_off"])[s["leaf"]]
        s["tgt_off"] = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        s["tgt_off"][1:] = per.cumsum(0)
        s["pair_tgt"] = torch.repeat_interleave(torch.arange(n, device=DEV), per)
        s["elem_idx"] = (torch.arange(s["pair_tgt"].numel(), device=DEV) - s["tgt_off"][s["pair_tgt"]]
                         + s["leaf_off"][s["leaf"][s["pair_tgt"]]])
    if op == "adjoint":
        s["grad"] = torch.randn(n_leaves, (c["p"] + 1) ** 2, dtype=torch.float64, device=DEV, generator=g)
    if op == "galerkin":
        s["weights"] = torch.randn(n_leaves, (c["p"] + 1) ** 2, dtype=torch.float64, device=DEV, generator=g)
    if op == "reduce":
        s["elem"] = _rows(g, n, c["p"], s["leaf_rho"][s["leaf"]])
    if op == "upward":
        s["coef"] = _rows(g, n_leaves, c["p"], s["leaf_rho"])
    return s


def _rows(g, n, p, rho, norm="coeff"):
    """Random coefficient rows with the size that coefficients about a centre
    have: rho^n / sqrt((n+m)! (n-m)!) at degree n, order m."""
    out = torch.randn(n, (p + 1) ** 2, dtype=torch.float64, device=DEV, generator=g)
    for deg in range(p + 1):
        f = [math.exp(-0.5 * (math.lgamma(deg + abs(m) + 1) + math.lgamma(deg - abs(m) + 1))) for m in range(-deg, deg + 1)]
        out[:, deg * deg:(deg + 1) ** 2] *= torch.tensor(f, dtype=torch.float64, device=DEV) * (rho ** deg)[:, None]
    return out


def _batch_inputs(c, g, mesh):
    """Three kinds of elements in one adaptive octree (a box is split while it
    holds more than max_leaf elements), with a degree per leaf."""
    kinds = {}
    v, el = _filaments(c["n_fil"], c["n_steps"], mesh)
    kinds["segments"] = (v, el, _uniform(g, el.shape[1]), 1e-4)
    v, el = _sphere(c["freq"], mesh)
    kinds["triangles"] = (0.9 * v, el, _uniform(g, el.shape[1]), 0.09 / c["freq"])
    v, el = _tets(c["grid"], mesh)
    kinds["tetra"] = (v, el, _uniform(g, el.shape[1], lo=0.0), 0.05 / c["grid"])
    deepest, lo, size = 12, -1.25, 2.5
    code = torch.cat([_cells(v, el, lo, size, deepest) for v, el, _, _ in kinds.values()])
    leaf_code = torch.full_like(code, -1)  # first deepest-level code of the element's leaf
    leaf_depth = torch.zeros_like(code)
    open_ = torch.ones_like(code, dtype=torch.bool)
    for d in range(deepest + 1):
        at = open_.nonzero()[:, 0]
        if not at.numel():
            break
        box = code[at] >> (3 * (deepest - d))
        _, inv, counts = torch.unique(box, return_inverse=True, return_counts=True)
        done = (counts[inv] <= c["max_leaf"]) | (d == deepest)
        sel = at[done]
        leaf_code[sel] = box[done] << (3 * (deepest - d))
        leaf_depth[sel] = d
        open_[sel] = False
    uniq, leaf = torch.unique(leaf_code, return_inverse=True)
    n_leaves = uniq.numel()
    depth = torch.zeros(n_leaves, dtype=torch.int64, device=DEV)
    depth[leaf] = leaf_depth
    h = size / (2.0 ** depth.double())
    corner = _unmorton(uniq, deepest).double() * (size / (1 << deepest))
    leaf_c = (lo + corner + 0.5 * h).contiguous()
    s, rho, base = dict(leaf_c=leaf_c, kinds={}), torch.zeros(n_leaves, dtype=torch.float64, device=DEV), 0
    for name, (v, el, sigma, amp) in kinds.items():
        v = _moved(v, g, amp)
        lk, order = torch.sort(leaf[base:base + el.shape[1]], stable=True)
        base += el.shape[1]
        el = el[:, order]
        off = torch.zeros(n_leaves + 1, dtype=torch.int64, device=DEV)
        off[1:] = torch.bincount(lk, minlength=n_leaves).cumsum(0)
        _leaf_rho(v, el, lk, leaf_c, rho)
        s["kinds"][name] = dict(vxyz=v, idx=el.to(torch.int32).contiguous(), sigma=sigma[order].contiguous(),
                                leaf_off=off, el=el, leaf=lk)
    s["leaf_rho"] = rho
    s["leaf_p"] = torch.randint(c["p_lo"], c["p_hi"] + 1, (n_leaves,), device=DEV, generator=g).to(torch.int32)
    return s


# ------------------------------------------------------------------- the call


def prepare(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    op = c["op"]
    if op == "adjoint":
        s["vxyz"].requires_grad_(True)
        s["sigma"].requires_grad_(True)
    norm = "moment" if op == "galerkin" else c.get("norm", "coeff")
    s["plan"] = q2x.Plan(c["p_hi"] if op == "batch" else c["p"] if "p" in c else 0, norm=norm,
                         precision=c.get("precision", "fp64"))
    if op == "batch":
        kinds = {k: {n: d[n] for n in ("vxyz", "idx", "sigma", "leaf_off")} for k, d in s["kinds"].items()}
        s["batch"] = Batch(s["plan"], s["leaf_c"], s["leaf_rho"], s["leaf_p"], tile_elems=512, **kinds)
    if op == "upward":
        s["upward"] = Upward(s["plan"], s["leaf_c"], s["lo"], s["width"], c["depth"])
    for k in ("el", "leaf", "pair_tgt", "kinds"):
        if not (k == "kinds" and op != "batch"):
            s.pop(k, None)
    s["case"] = c
    return s


def run(s):
    c, plan = s["case"], s["plan"]
    op = c["op"]
    if op == "elements":
        rho = s["leaf_rho"] if c["rho"] else None
        args = (s["vxyz"], s["idx"], s["sigma"], s["leaf_off"], s["leaf_c"], rho, s["leaf_p"])
        if c["kind"] == "segment":
            return plan.segments(*args)
        if c["kind"] == "tetra":
            return plan.tetra(*args)
        return plan.triangles(*args, density=c["density"], single=c["single"], double=c["double"])
    if op == "batch":
        return s["batch"].run()
    if op == "adjoint":
        coef = triangles_single(s["vxyz"], s["sigma"], plan, s["idx"], s["leaf_off"], s["leaf_c"], s["leaf_rho"])
        gv, gs = torch.autograd.grad(coef, (s["vxyz"], s["sigma"]), s["grad"])
        return coef.detach(), gv, gs
    if op == "currents":
        coef3 = plan.segments_vector(s["vxyz"], s["idx"], s["current"], s["leaf_off"], s["leaf_c"], s["leaf_rho"])
        return coef3, plan.evaluate_curl(s["coef"], s["exp_c"], s["tgt"], s["tgt_off"], s["exp_idx"])
    if op == "upward":
        return s["upward"].run(s["coef"])
    if op == "far":
        return plan.evaluate(s["coef"][0], s["exp_c"], s["tgt"], s["tgt_off"], s["exp_idx"])
    if op == "near":
        return plan.nearfield(c["kind"], s["vxyz"], s["idx"], s["sigma"], s["tgt"], s["tgt_off"], s["elem_idx"],
                              layer=c["layer"])
    if op == "galerkin":
        return plan.galerkin_triangles(s["vxyz"], s["idx"], s["weights"], s["leaf_off"], s["leaf_c"], s["leaf_rho"],
                                       s["sigma"], layer=c["layer"])
    return plan.leaf_reduce(s["elem"], c["p"], s["leaf_off"])


# ------------------------------------------------------------------- the work


def _leaves_of(n, depth, surface):
    """About how many leaves a uniform octree has (the closed surface's area, the filaments' volume)."""
    return max(1.0, min(float(n), (3.65 * 4.0 ** depth) if surface else 0.3 * 8.0 ** depth))


def work(case):
    c = dict(case)
    op, p = c["op"], c.get("p", c.get("p_hi", 0))
    np_ = (p + 1) ** 2
    entries = (p + 1) * (p + 2) / 2  # complex (n, m >= 0)

    def element(kind, density="const", both=False):
        levels = NV[kind] - 1 + (2 if density == "linear" else 0)
        # a level's three-term complex step a (n, m): 16 operations; the leaf sum: one a coefficient
        return (7 + 16.0 * levels + (16 if both else 0)) * entries + np_ * (2 if both else 1)

    def element_bytes(kind, n):
        return n * (4 * NV[kind] + 8 + 12)

    if op == "elements":
        n = _count(c["kind"], c["size"])
        layers = int(c["single"]) + int(c["double"])
        nl = _leaves_of(n, c["depth"], c["kind"] != "tetra")
        return dict(bytes=element_bytes(c["kind"], n) + nl * (40 + 8 * np_ * layers),
                    flops=n * element(c["kind"], c["density"], layers == 2))
    if op == "batch":
        seg, tri, tet = c["n_fil"] * c["n_steps"], 20 * c["freq"] ** 2, 6 * c["grid"] ** 3
        nl = (seg + tri + tet) / (0.3 * c["max_leaf"])
        mean = 0.7  # of the largest degree's work, over the degrees of the leaves
        return dict(bytes=element_bytes("segment", seg) + element_bytes("triangle", tri) + element_bytes("tetra", tet)
                    + nl * 8 * np_,
                    flops=mean * (seg * element("segment") + tri * element("triangle") + tet * element("tetra")))
    if op == "currents":
        n = c["n_fil"] * c["n_steps"]
        nl = _leaves_of(n, c["depth"], False)
        return dict(bytes=element_bytes("segment", n) + 16 * n + nl * (40 + 24 * np_) + c["n_tgt"] * 56,
                    flops=n * (element("segment") + 6 * np_) + c["n_tgt"] * entries * 50.0)
    if op == "far":
        m = c["n_tgt"] * c["per_target"]
        return dict(bytes=c["n_exp"] * 8 * (np_ + 3) + c["n_tgt"] * 40 + 8 * m, flops=m * 9.0 * entries)
    n = 20 * c["freq"] ** 2
    nl = _leaves_of(n, c["depth"], True)
    if op == "adjoint":
        return dict(bytes=2 * element_bytes("triangle", n) + nl * (40 + 16 * np_) + n * 20,
                    flops=n * (element("triangle") + (7 * 16.0 + 40) * entries))
    if op == "upward":
        return dict(bytes=1.35 * nl * 8 * np_, flops=1.35 * nl * 8.0 * (p + 1) ** 4 / 8)
    if op == "near":
        m = n * n / nl * 1.4
        return dict(bytes=element_bytes(c["kind"], n) + 40 * n + 8 * m, flops=m * (105.0 if c["kind"] == "triangle" else 40.0))
    if op == "galerkin":
        return dict(bytes=element_bytes("triangle", n) + nl * (40 + 8 * np_) + 8 * n, flops=n * (element("triangle") + np_))
    return dict(bytes=8.0 * np_ * (n + nl), flops=float(n * np_))


# ----------------------------------------------------- the outputs in 64 bits
#
# Tilde recursions of the paper's Lemmas 1-5 as complex torch arithmetic,
# all elements at once: rows (orders 0..n, elements), one level after another.


def _stencil(a, xi, eta, z, n):
    """-xi a^{m-1} + eta a^{m+1} - z a^m for orders 0..n of the row `a` of degree n - 1."""
    out = torch.zeros(n + 1, xi.shape[0], dtype=torch.complex128, device=xi.device)
    if n == 0:
        return out
    out = out.clone()
    out[:n] = out[:n] - z * a
    out[1:] = out[1:] - xi * a
    if n > 1:
        out[1:n - 1] = out[1:n - 1] + eta * a[2:]
        out[0] = out[0] + 2.0 * (eta * a[1]).real
    return out


def _point(x):
    xi = torch.complex(0.5 * x[0], 0.5 * x[1])
    return xi, xi.conj(), x[2]


def _moments(kind, X, p, sig=None, normal=None):
    """Rows 0..p of the element integrals over the unit simplex (without the
    Jacobian) of the vertices X (one (3, n) tensor a vertex about the centre);
    with `sig` (the three vertex densities) the density's; with `normal` the
    normal derivative's as well. Yields (n, single row, double row)."""
    V = [_point(x) for x in X]
    order = {"segment": [1, 0], "triangle": [1, 2, 0], "tetra": [1, 2, 3, 0]}[kind]
    rows = [None] * len(order)
    E = W = None
    nu = _point(normal) if normal is not None else None
    for n in range(p + 1):
        last = W if sig is not None else rows[-1]
        dbl = _stencil(last, *nu, n) if nu is not None else None
        new = []
        for k, v in enumerate(order):
            if n == 0:
                r = torch.full((1, X[0].shape[1]), 1.0 / math.factorial(k), dtype=torch.complex128, device=X[0].device)
            else:
                r = _stencil(rows[k], *V[v], n)
                r = (r + new[k - 1]) / (n + k) if k else r / n
            new.append(r)
        if sig is not None:
            s1, s2, s3 = sig
            q, j, i = new
            e = (0.0 if n == 0 else _stencil(E, *V[2], n)) + s2 * q + s3 * j
            E2 = e / (n + 2)
            w = (0.0 if n == 0 else _stencil(W, *V[0], n)) + E2 + s1 * i
            E, W = E2, w / (n + 3)
        rows = new
        yield n, (W if sig is not None else rows[-1]), dbl


def _packed(row, n, norm):
    """The packed real columns of degree n (2n + 1, elements), without the Jacobian."""
    m = torch.arange(n + 1, device=row.device)
    phase = torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device=row.device)
    if norm == "coeff":
        f = (phase[m % 4] * ((-1.0) ** (n + m)) / (4 * math.pi))[:, None] * row.conj()
    else:
        f = phase[(-m) % 4][:, None] * row
    return torch.cat([f[1:].imag.flip(0), f.real])


def _jacobian(X):
    e = [x - X[0] for x in X[1:]]
    if len(e) == 1:
        return e[0].norm(dim=0)
    cr = torch.linalg.cross(e[0], e[1], dim=0)
    return cr.norm(dim=0) if len(e) == 2 else (cr * e[2]).sum(0).abs()


def _chunks(n, size=131072):
    return [(a, min(n, a + size)) for a in range(0, n, size)]


def _sums(kind, s, p, norm="coeff", density="const", single=True, double=False, weights=None, out=None):
    """Leaf coefficients of one kind: [single, double] (weights: one output a weight row)."""
    el, leaf, v = s["el"], s["leaf"], s["vxyz"].detach()
    n_leaves = s["n_leaves"] if "n_leaves" in s else s["leaf_c"].shape[1]
    n_out = weights.shape[0] if weights is not None else 2
    if out is None:
        out = [torch.zeros((p + 1) ** 2, n_leaves, dtype=torch.float64, device=DEV) if w else None
               for w in ([True] * n_out if weights is not None else (single, double))]
    for a, b in _chunks(el.shape[1]):
        lf = leaf[a:b]
        V = [v[:, el[k, a:b]] for k in range(el.shape[0])]  # edges from the vertices as given
        X = [x - s["leaf_c"][:, lf] for x in V]
        J = _jacobian(V)
        normal = None
        if double:
            cr = torch.linalg.cross(V[1] - V[0], V[2] - V[0], dim=0)
            normal = cr / cr.norm(dim=0)
        sig = [s["sigma"].detach()[el[k, a:b]] for k in range(3)] if density == "linear" else None
        dens = [J] if sig else [J * w[a:b] for w in (weights if weights is not None else [s["sigma"].detach()])]
        for n, r, d in _moments(kind, X, p, sig, normal):
            at = slice(n * n, (n + 1) ** 2)
            for o, (rows, w) in enumerate([(r, w) for w in dens] if weights is not None else [(r, dens[0]), (d, dens[0])]):
                if out[o] is not None and rows is not None:
                    out[o][at].index_add_(1, lf, _packed(rows, n, norm) * w)
    return out


def _cut(rows, leaf_p, p):
    if leaf_p is not None:
        deg = torch.cat([torch.full((2 * n + 1,), n, device=DEV) for n in range(p + 1)])
        rows = rows * (deg[:, None] <= leaf_p[None])
    return rows.t().contiguous()


def _singular(p, x):
    """S_n^m (m >= 0) at offsets x (3, n): a list over the degrees of complex (n + 1, targets)."""
    r2 = (x * x).sum(0)
    xy = torch.complex(x[0], x[1])
    cols, tmm = [], torch.ones_like(xy)
    for m in range(p + 1):
        if m:
            tmm = -(2 * m - 1) * xy * tmm
        col = [tmm]
        if m < p:
            col.append((2 * m + 1) * x[2] * tmm)
        for n in range(m + 2, p + 1):
            col.append(((2 * n - 1) * x[2] * col[-1] - (n + m - 1) * r2 * col[-2]) / (n - m))
        cols.append(col)
    inv = r2.sqrt()
    return [torch.stack([cols[m][n - m] * ((1j) ** (-m % 4) if m % 4 else 1.0) * math.factorial(n - m) / inv ** (2 * n + 1)
                         for m in range(n + 1)]) for n in range(p + 1)]


def _potential(F, p, norm, x):
    """sum F_n^m S_n^m of one row (p + 1)^2 a target, F (columns, targets) or (columns, 1)."""
    tot = 0.0
    for n, S in enumerate(_singular(p, x)):
        k = n * n + n
        for m in range(n + 1):
            re, im = F[k + m], (F[k - m] if m else torch.zeros_like(F[k]))
            if norm == "moment":
                sgn = (-1.0) ** (n + m) / (4 * math.pi)
                re, im = sgn * re, -sgn * im
            t = re * S[m].real - im * S[m].imag
            tot = tot + (2.0 * t if m else t)
    return tot


def _log_piece(sm, sp, Rm, Rp, d2, length):
    """log((Rp + sp) / (Rm + sm)) without cancellation, as log1p of the exactly rearranged ratio."""
    tot, s = Rm + Rp, sm + sp
    ahead = s >= 0
    near = torch.where(ahead, Rm, Rp)
    at = torch.where(ahead, sm, -sp)
    den = torch.where(at >= 0, near + at, d2 / (near - at))
    return torch.log1p(length * (tot + s.abs()) / (tot * den))


def _triangle_pairs(r, X, layer):
    """Single layer integral of 1/R, or double layer's solid angle, of triangles X at targets r (pairs)."""
    cr = torch.linalg.cross(X[1] - X[0], X[2] - X[0], dim=0)
    J = cr.norm(dim=0)
    n = cr / J
    h = ((r - X[0]) * n).sum(0)
    snap = 16 * 2.220446049250313e-16 * (r.abs().sum(0) + X[0].abs().sum(0))  # targets in the plane, as documented
    h = torch.where(h.abs() <= snap, torch.zeros_like(h), h)
    R = [(x - r).norm(dim=0) for x in X]
    d = [x - r for x in X]
    den = (R[0] * R[1] * R[2] + (d[0] * d[1]).sum(0) * R[2] + (d[0] * d[2]).sum(0) * R[1] + (d[1] * d[2]).sum(0) * R[0])
    solid = torch.where(h == 0, torch.zeros_like(h), 2.0 * torch.atan2(J * h, den))
    if layer:
        return solid
    tot = -h * solid
    for k in range(3):
        e = X[(k + 1) % 3] - X[k]
        length = e.norm(dim=0)
        l = e / length
        t = (d[k] * torch.linalg.cross(l, n, dim=0)).sum(0)
        t = torch.where(t.abs() <= snap, torch.zeros_like(t), t)
        log = _log_piece((d[k] * l).sum(0), (d[(k + 1) % 3] * l).sum(0), R[k], R[(k + 1) % 3], t * t + h * h, length)
        tot = tot + torch.where(t == 0, torch.zeros_like(t), t * log)
    return tot


def _translation_matrix(t, p):
    """Real (columns, columns) matrix of coefficients about c moved to c - t (COEFF norm)."""
    R = {(0, 0): 1.0 + 0j}
    ix, ie = 1j * (t[0] + 1j * t[1]) / 2, 1j * (t[0] - 1j * t[1]) / 2
    for n in range(1, p + 1):
        for m in range(-n, n + 1):
            R[n, m] = (ix * R.get((n - 1, m - 1), 0) + ie * R.get((n - 1, m + 1), 0) - t[2] * R.get((n - 1, m), 0)) / n
    M = np.zeros(((p + 1) ** 2, (p + 1) ** 2))
    for n in range(p + 1):
        for m in range(n + 1):
            for k in range(n + 1):
                for l in range(-k, k + 1):
                    nn, mm = n - k, m + l
                    if abs(mm) > nn:
                        continue
                    c = (-1) ** k * R[k, l]
                    a, sg = abs(mm), 1.0
                    cj = mm < 0  # F^{-a} = (-1)^a conj F^a
                    if cj:
                        c = c * (-1) ** a
                    ko, ks = n * n + n, nn * nn + nn
                    sg = -1.0 if cj else 1.0
                    M[ko + m, ks + a] += c.real
                    if a:
                        M[ko + m, ks - a] -= sg * c.imag
                    if m:
                        M[ko - m, ks + a] += c.imag
                        if a:
                            M[ko - m, ks - a] += sg * c.real
    return torch.from_numpy(M).to(DEV)


def exact(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    op, p = c["op"], c.get("p", c.get("p_hi", 0))
    if op == "elements":
        outs = _sums(c["kind"], s, p, c["norm"], c["density"], c["single"], c["double"])
        outs = [None if o is None else _cut(o, s["leaf_p"], p) for o in outs]
        return outs if c["kind"] == "triangle" else outs[0]
    if op == "batch":
        out = None
        for name, d in s["kinds"].items():
            out = _sums({"segments": "segment", "triangles": "triangle", "tetra": "tetra"}[name],
                        dict(d, leaf_c=s["leaf_c"]), p, out=out, single=True)
        return _cut(out[0], s["leaf_p"], p)
    if op == "adjoint":
        coef = _sums("triangle", s, p)[0].t().contiguous()
        el, v = s["el"], s["vxyz"]
        gv, gs = torch.zeros_like(v), torch.zeros_like(s["sigma"])
        for a, b in _chunks(el.shape[1], 32768):
            lf = s["leaf"][a:b]
            V = [v[:, el[k, a:b]].requires_grad_(True) for k in range(3)]
            X = [x - s["leaf_c"][:, lf] for x in V]
            sg = s["sigma"][a:b].clone().requires_grad_(True)
            J = _jacobian(V)
            loss = 0.0
            for n, r, _ in _moments("triangle", X, p):
                loss = loss + (_packed(r, n, "coeff") * (J * sg) * s["grad"].t()[n * n:(n + 1) ** 2, lf]).sum()
            got = torch.autograd.grad(loss, V + [sg])
            for k in range(3):
                gv.index_add_(1, el[k, a:b], got[k])
            gs[a:b] = got[3]
        return coef, gv, gs
    if op == "currents":
        coef3 = torch.stack([o.t() for o in _sums("segment", s, p, weights=s["current"])])
        H = torch.zeros(3, c["n_tgt"], dtype=torch.float64, device=DEV)
        for a, b in _chunks(c["n_tgt"], 32768):
            x = (s["tgt"][:, a:b] - s["exp_c"]).requires_grad_(True)
            g = [torch.autograd.grad(_potential(s["coef"][k].t(), p, "coeff", x).sum(), x)[0] for k in range(3)]
            H[0, a:b], H[1, a:b], H[2, a:b] = g[2][1] - g[1][2], g[0][2] - g[2][0], g[1][0] - g[0][1]
        return coef3, H
    if op == "far":
        out = torch.zeros(c["n_tgt"], dtype=torch.float64, device=DEV)
        idx = s["exp_idx"].reshape(c["n_tgt"], c["per_target"])
        for a, b in _chunks(c["n_tgt"], 65536):
            for k in range(c["per_target"]):
                e = idx[a:b, k]
                F = s["coef"][0].t() if c["n_exp"] == 1 else s["coef"][0][e].t()
                out[a:b] += _potential(F, p, c["norm"], s["tgt"][:, a:b] - s["exp_c"][:, e])
        return out
    if op == "near":
        out = torch.zeros(s["tgt"].shape[1], dtype=torch.float64, device=DEV)
        for a, b in _chunks(s["elem_idx"].numel(), 2097152):
            e, t = s["elem_idx"][a:b], s["pair_tgt"][a:b]
            r = s["tgt"][:, t]
            X = [s["vxyz"][:, s["el"][k, e]] for k in range(s["el"].shape[0])]
            if c["kind"] == "triangle":
                val = _triangle_pairs(r, X, c["layer"])
            else:
                ev = X[1] - X[0]
                length = ev.norm(dim=0)
                l = ev / length
                pa, pb = X[0] - r, X[1] - r
                d2 = (torch.linalg.cross(pa, l, dim=0) ** 2).sum(0)
                val = _log_piece((pa * l).sum(0), (pb * l).sum(0), pa.norm(dim=0), pb.norm(dim=0), d2, length)
            out.index_add_(0, t, s["sigma"][e] * val / (4 * math.pi))
        return out
    if op == "galerkin":
        el, out = s["el"], torch.zeros(s["el"].shape[1], dtype=torch.float64, device=DEV)
        for a, b in _chunks(el.shape[1]):
            lf = s["leaf"][a:b]
            V = [s["vxyz"][:, el[k, a:b]] for k in range(3)]
            X = [x - s["leaf_c"][:, lf] for x in V]
            cr = torch.linalg.cross(V[1] - V[0], V[2] - V[0], dim=0)
            normal = cr / cr.norm(dim=0) if c["layer"] else None
            w = s["weights"].t()[:, lf]
            for n, r, d in _moments("triangle", X, p, None, normal):
                out[a:b] += (_packed(d if c["layer"] else r, n, "moment") * w[n * n:(n + 1) ** 2]).sum(0)
            out[a:b] *= _jacobian(V) * s["sigma"][a:b]
        return out
    if op == "reduce":
        out = torch.zeros(s["leaf_c"].shape[1], (p + 1) ** 2, dtype=torch.float64, device=DEV)
        return out.index_add_(0, s["leaf"], s["elem"])
    # upward: level by level, the translations of one shift as one matrix product
    coef, depth, h = s["coef"], c["depth"], s["width"] / (1 << c["depth"])
    code = _morton(((s["leaf_c"] - s["lo"]) / h).floor().to(torch.int64), depth)
    outs = []
    for d in range(depth - 1, -1, -1):
        uniq, parent = torch.unique_consecutive(code >> 3, return_inverse=True)
        out = torch.zeros(uniq.numel(), coef.shape[1], dtype=torch.float64, device=DEV)
        for child in range(8):
            sel = (code & 7) == child
            half = s["width"] / (1 << d) / 4
            t = [half * (2 * ((child >> (2 - k)) & 1) - 1) for k in range(3)]
            if bool(sel.any()):
                out.index_add_(0, parent[sel], coef[sel] @ _translation_matrix(t, p).t())
        outs.append(out)
        coef, code = out, uniq
    return outs
