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
from _helpers import random_problem

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
    """(leaf sums, per-element rows summed in leaves, the sums of the magnitudes
    of the rows for densities |sigma|), each a list over the layers."""
    import torch
    plan = q2x.Plan(p, norm=norm)
    off = prob["leaf_off"]
    leaf_of = np.repeat(np.arange(len(off) - 1), np.diff(off))
    got = call(plan, prob, off, prob["leaf_c"], prob["leaf_rho"] if rho else None, prob["leaf_p"], layers)
    rows = call(plan, prob, None, prob["leaf_c"][:, leaf_of], prob["leaf_rho"][leaf_of] if rho else None,
                prob["leaf_p"][leaf_of], layers)
    off_d = torch.from_numpy(off).cuda()
    ref = [None if r is None else plan.leaf_reduce(r, p, off_d) for r in rows]
    rows = call(plan, dict(prob, sigma=np.abs(prob["sigma"])), None, prob["leaf_c"][:, leaf_of],
                prob["leaf_rho"][leaf_of] if rho else None, prob["leaf_p"][leaf_of], layers)
    size = [None if r is None else plan.leaf_reduce(r.abs(), p, off_d) for r in rows]
    plan.sync()
    return got, ref, size


def check(prob, p, got, ref, size):
    """_helpers.norm_err of all leaves at once, against the largest sum of
    magnitudes: a leaf of one or two elements can cancel in its own sums."""
    for layer, (g, r, z) in enumerate(zip(got, ref, size)):
        if r is not None:
            n = _degree(p)
            f = _scales(p) / (np.maximum(n, 1.0) if layer else 1.0)
            s = f / prob["leaf_rho"][:, None] ** (np.maximum(n - 1, 0) if layer else n)
            a, b = g.cpu().numpy() * s, r.cpu().numpy() * s
            top = (z.cpu().numpy() * s).max(axis=1)
            assert np.all(np.abs(a - b).max(axis=1) <= 1e-12 * np.where(top > 0, top, 1.0))


def edge_sizes(p, case):
    """Leaf sizes about the edges of a group, a full tile and two tiles for the
    CTA sizes of small leaves (64, 128 threads, among thousands of tiny leaves)
    or of large ones (128 to 256, among leaves of 700); "few": the latter alone,
    too few elements for full tiles on every SM."""
    sizes = [1, 0, 2, 7, 8, 9, 33]
    for nt in (64, 128) if case == "small" else (128, 160, 192, 256):
        groups = max(1, nt // (p + 1))
        full = min(8 * groups, nt)
        sizes += [max(groups - 1, 1), groups, groups + 1, full - 1, full, full + 1, 0, min(2 * full + 1, 600)]
    return sizes + {"small": [1, 2, 3, 1, 0, 5] * 900, "large": [700] * 60, "few": [500]}[case]


@pytest.mark.parametrize("kind,density", KINDS)
@pytest.mark.parametrize("case", ["few", "small", "large"])
@pytest.mark.parametrize("p", [0, 1, 2, 5, 11, 13, 15, 18, 20])
def test_tile_edges(q2x, kind, density, p, case):
    prob = random_problem(kind, edge_sizes(p, case), seed=p + 50, p=p, density=density)
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
    base = both(q2x, prob, p, (True, False))[0]
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
    assert np.array_equal(np.isfinite(got), np.isfinite(want))  # beyond FP64 in both (tiles of both signs: NaN)


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


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n_leaves,p", [(1, 3), (3, 20), (1023, 9), (1024, 3), (1025, 3), (12000, 9), (100000, 9)])
def test_tile_list_and_offset_check(q2x, n_leaves, p, precision):
    """The tile list's one-block build and the general one about their border,
    and the combine with one to 32 leaves and all or fewer columns a warp:
    empty leaves at both ends, some of many tiles, the same sums as the
    per-element rows, and bad offsets reported."""
    rng = np.random.default_rng(n_leaves)
    sizes = rng.integers(0, 4, n_leaves)
    sizes[[0, -1]] = 0
    sizes[n_leaves // 2] = 2000
    sizes[n_leaves // 3::999] = 300
    prob = random_problem("segment", list(sizes), seed=5, p=p)
    plan = q2x.Plan(p, precision=precision)
    got = call(plan, prob, prob["leaf_off"], prob["leaf_c"], prob["leaf_rho"], prob["leaf_p"], (True,))[0]
    if precision == "fp64":
        check(prob, p, [got], *both(q2x, prob, p, (True,))[1:])
    assert plan.device_errors() == 0
    for at, v in ((0, 1), (n_leaves, int(sizes.sum()) - 1), (n_leaves // 2, int(sizes.sum()) + 5)):
        off = prob["leaf_off"].copy()
        off[at] = v
        call(plan, prob, off, prob["leaf_c"], prob["leaf_rho"], prob["leaf_p"], (True,))
        assert plan.device_errors() & 8


@pytest.mark.parametrize("p", [0, 1, 6, 12, 16, 20])
def test_vector_density(q2x, p):
    """The three components of a line current, at tile edges, with a component that vanishes and one far smaller than the others."""
    import torch
    prob = random_problem("segment", edge_sizes(p, "large"), seed=p + 9, p=p)
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
@pytest.mark.parametrize("case", ["few", "small", "large"])
@pytest.mark.parametrize("p", [0, 1, 4, 12, 17, 20])
def test_galerkin_side(q2x, p, case, layer):
    """Receiver-side integrals against per-element rows contracted on the host,
    weights of all degrees of one size in the scaled norm."""
    import torch
    prob = random_problem("triangle", edge_sizes(p, case), seed=p + 70, p=p)
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
