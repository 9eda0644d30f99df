"""The FP64 leaf sums by directions (csrc/q2x_dir.cuh) at the sizes where their
tiling and number format could go wrong: tiles that are just full, just over
and nearly empty, every kind and layer at degrees between the tested bins,
coordinates in other units, and very uneven weights.  Reference: the same
library's per-element rows (the FP64 row kernel, another algorithm), summed in
leaves by q2x_leaf_reduce.

Tolerance: both paths round each element's moments to a few units of 2^-53 of
its own scale, and a leaf of K elements sums K of them; with K <= 700 and the
scaled norm of _helpers (degree n over rho^n) 1e-12 is the suite's FP64 bound."""
import numpy as np
import pytest
from _helpers import norm_err, random_problem

pytestmark = pytest.mark.gpu
KINDS = [("segment", "const"), ("triangle", "const"), ("triangle", "linear"), ("tetra", "const")]


@pytest.fixture(scope="module")
def q2x():
    import paper_2107_10942_gb300 as q
    return q


def call(plan, prob, off, c, rho, lp, layers):
    import torch
    d = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in prob.items() if hasattr(v, "dtype")}
    t = [None if x is None else torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (off, c, rho, lp)]
    args = (d["vxyz"], d["idx"], d["sigma"], *t)
    if prob["kind"] == "segment":
        return [plan.segments(*args)]
    if prob["kind"] == "tetra":
        return [plan.tetra(*args)]
    return list(plan.triangles(*args, density=prob["density"], single=layers[0], double=layers[1]))


def both(q2x, prob, p, layers, rho=True, norm="coeff"):
    """(leaf sums, per-element rows summed in leaves), each a list over the layers."""
    import torch
    plan = q2x.Plan(p, norm=norm)
    off = prob["leaf_off"]
    leaf_of = np.repeat(np.arange(len(off) - 1), np.diff(off))
    got = call(plan, prob, off, prob["leaf_c"], prob["leaf_rho"] if rho else None, prob["leaf_p"], layers)
    rows = call(plan, prob, None, prob["leaf_c"][:, leaf_of], prob["leaf_rho"][leaf_of] if rho else None,
                prob["leaf_p"][leaf_of], layers)
    off_d = torch.from_numpy(off).cuda()
    ref = [None if r is None else plan.leaf_reduce(r, p, off_d) for r in rows]
    plan.sync()
    return got, ref


def check(prob, p, got, ref):
    for layer, (g, r) in enumerate(zip(got, ref)):
        if r is not None:
            assert norm_err(g.cpu().numpy(), r.cpu().numpy(), p, prob["leaf_rho"], layer) <= 1e-12


def edge_sizes(p, small):
    """Leaf sizes about the edges of a group, a full tile and two tiles for the
    CTA sizes of small leaves (64, 128 threads; many tiny leaves among them) or
    of large ones (128 to 256)."""
    sizes = [1, 0, 2, 7, 8, 9, 33]
    for nt in (64, 128) if small else (128, 160, 192, 256):
        groups = max(1, nt // (p + 1))
        full = min(8 * groups, nt)
        sizes += [max(groups - 1, 1), groups, groups + 1, full - 1, full, full + 1, 0, min(2 * full + 1, 600)]
    return sizes + ([1, 2, 3, 1, 0, 5] * 40 if small else [500, 700])


@pytest.mark.parametrize("kind,density", KINDS)
@pytest.mark.parametrize("small", [True, False])
@pytest.mark.parametrize("p", [0, 1, 2, 5, 11, 13, 15, 18, 20])
def test_tile_edges(q2x, kind, density, p, small):
    prob = random_problem(kind, edge_sizes(p, small), seed=p + 50, p=p, density=density)
    layers = (True, kind == "triangle")
    check(prob, p, *both(q2x, prob, p, layers))


@pytest.mark.parametrize("layers", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("density", ["const", "linear"])
def test_layers_and_ragged_degrees(q2x, layers, density):
    p, sizes = 17, [5, 120, 121, 1, 64]
    prob = random_problem("triangle", sizes, seed=3, p=p, density=density, leaf_p=[17, 3, 16, 0, 9])
    check(prob, p, *both(q2x, prob, p, layers, norm="moment"))


@pytest.mark.parametrize("unit", [1e-140, 1e-30, 3.7, 1e25, 1e90])
@pytest.mark.parametrize("kind,density", KINDS)
def test_units(q2x, kind, density, unit):
    """Coordinates in another unit scale degree n of a kind of dimension d by
    unit^(n + d) (single layer); p = 2 keeps that inside FP64 at these units."""
    p = 2
    prob = random_problem(kind, [9, 40, 3], seed=8, p=p, density=density)
    base, _ = both(q2x, prob, p, (True, False))
    for k in ("vxyz", "leaf_c", "leaf_rho"):
        prob[k] = prob[k] * unit
    got = both(q2x, prob, p, (True, False), rho=False)[0][0].cpu().numpy()
    dim = {"segment": 1, "triangle": 2, "tetra": 3}[kind]
    scale = np.concatenate([np.full(2 * n + 1, float(n + dim)) for n in range(p + 1)])
    with np.errstate(over="ignore", under="ignore"):
        want = base[0].cpu().numpy() * unit ** scale
    ok = (np.abs(want) > 1e-290) & np.isfinite(want)
    # the scaled coordinates themselves are rounded: up to (p + 1) units of 2^-53 of the leaf's largest
    for n in range(p + 1):
        cols = slice(n * n, (n + 1) ** 2)
        big = np.max(np.abs(np.where(ok, want, 0.0))[:, cols], axis=1, keepdims=True)
        diff = np.abs(np.where(ok, got, 0.0) - np.where(ok, want, 0.0))[:, cols]
        assert np.all(diff <= 1e-12 * big + 1e-290)
    assert np.array_equal(np.isinf(got), np.isinf(want))  # beyond FP64 in both


def test_uneven_weights(q2x):
    """A heavy element beside light ones, and elements of no weight far out: the
    sums stay relative to the leaf's largest term."""
    p = 12
    prob = random_problem("triangle", [50, 50], seed=4, p=p)
    prob["sigma"][:25] *= 1e-9
    prob["sigma"][60:] = 0.0
    check(prob, p, *both(q2x, prob, p, (True, True)))


def test_accumulate_and_repeat(q2x):
    """Accumulation into leaves of one and of several tiles, and bit equality of repeated calls."""
    import torch
    p = 9
    prob = random_problem("triangle", [0, 3, 700, 90], seed=6, p=p)
    plan = q2x.Plan(p)
    d = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in prob.items() if hasattr(v, "dtype")}
    args = (d["vxyz"], d["idx"], d["sigma"], d["leaf_off"], d["leaf_c"], d["leaf_rho"], d["leaf_p"])
    one, _ = plan.triangles(*args)
    again, _ = plan.triangles(*args)
    assert torch.equal(one, again)
    base = torch.rand_like(one)
    acc = base.clone()
    plan.triangles(*args, coef_single=acc, accumulate=True)
    assert torch.equal(acc, base + one)


@pytest.mark.parametrize("p", [0, 1, 6, 12, 16, 20])
def test_vector_density(q2x, p):
    """The three components of a line current, at tile edges, with a component that vanishes and one far smaller than the others."""
    import torch
    prob = random_problem("segment", edge_sizes(p, False), seed=p + 9, p=p)
    rng = np.random.default_rng(p)
    cur = rng.uniform(-1, 1, size=(3, prob["idx"].shape[1]))
    cur[1, :60] = 0.0
    cur[2] *= 1e-6
    d = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in dict(prob, cur=cur).items() if hasattr(v, "dtype")}
    plan = q2x.Plan(p)
    got = plan.segments_vector(d["vxyz"], d["idx"], d["cur"], d["leaf_off"], d["leaf_c"], d["leaf_rho"], d["leaf_p"])
    base = torch.rand_like(got)
    acc = base.clone()
    plan.segments_vector(d["vxyz"], d["idx"], d["cur"], d["leaf_off"], d["leaf_c"], d["leaf_rho"], d["leaf_p"],
                         coef3=acc, accumulate=True)
    assert torch.equal(acc, base + got)
    one = torch.ones_like(d["sigma"])
    leaf_of = np.repeat(np.arange(len(prob["leaf_off"]) - 1), np.diff(prob["leaf_off"]))
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    rows = plan.segments(d["vxyz"], d["idx"], one, None, t(prob["leaf_c"][:, leaf_of]), t(prob["leaf_rho"][leaf_of]))
    ref = plan.leaf_reduce_weighted(rows, p, d["leaf_off"], d["cur"]).cpu().numpy()
    plan.sync()
    # the components share one scale, the largest current of the leaf: errors
    # against the largest coefficient of the degree over the three components
    top = _degree_max(np.abs(ref).max(axis=0), p)
    for k in range(3):
        assert np.all(np.abs(got[k].cpu().numpy() - ref[k]) <= 1e-12 * np.maximum(top, 1e-300)), k


def _degree_max(a, p):
    """Per leaf and column, the largest magnitude over the column's degree."""
    out = np.zeros_like(a)
    for n in range(p + 1):
        out[:, n * n:(n + 1) ** 2] = a[:, n * n:(n + 1) ** 2].max(axis=1, keepdims=True)
    return out


@pytest.mark.parametrize("layer", [0, 1])
@pytest.mark.parametrize("small", [True, False])
@pytest.mark.parametrize("p", [0, 1, 4, 12, 17, 20])
def test_galerkin_side(q2x, p, small, layer):
    """Receiver-side integrals against per-element rows contracted on the host,
    weights of all degrees of one size in the scaled norm."""
    import torch
    prob = random_problem("triangle", edge_sizes(p, small), seed=p + 70, p=p)
    rng = np.random.default_rng(p)
    leaf_of = np.repeat(np.arange(len(prob["leaf_off"]) - 1), np.diff(prob["leaf_off"]))
    w = rng.standard_normal((prob["leaf_c"].shape[1], (p + 1) ** 2)) * _scales(p) / prob["leaf_rho"][:, None] ** _degree(p)
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    d = {k: t(v) for k, v in prob.items() if hasattr(v, "dtype")}
    plan = q2x.Plan(p, norm="moment")
    got = plan.galerkin_triangles(d["vxyz"], d["idx"], t(w), d["leaf_off"], d["leaf_c"], d["leaf_rho"], d["sigma"],
                                  layer=layer).cpu().numpy()
    rows = plan.triangles(d["vxyz"], d["idx"], d["sigma"], None, t(prob["leaf_c"][:, leaf_of]),
                          t(prob["leaf_rho"][leaf_of]), single=layer == 0, double=layer == 1)[layer].cpu().numpy()
    plan.sync()
    terms = rows * w[leaf_of]
    # both sides round every column's term to some (p + 1) units of 2^-53 of its bound: the
    # degree's largest weight times the element's largest scaled row entry, 2n + 1 columns
    size = np.abs(w * prob["leaf_rho"][:, None] ** _degree(p) / _scales(p)).max(1)[leaf_of] * np.abs(
        rows / prob["leaf_rho"][leaf_of][:, None] ** _degree(p) * _scales(p)).max(1)
    assert np.all(np.abs(got - terms.sum(1)) <= 1e-13 * (p + 1) ** 2 * np.maximum(size, 1e-300))


def _degree(p):
    return np.concatenate([np.full(2 * n + 1, float(n)) for n in range(p + 1)])


def _scales(p):
    import math
    return np.array([math.sqrt(math.factorial(n + abs(m)) * math.factorial(n - abs(m)))
                     for n in range(p + 1) for m in range(-n, n + 1)])
