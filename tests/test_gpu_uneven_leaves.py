"""FP64 results by directions (csrc/q2x_dir.cuh) where the elements of a leaf
are very unequal: every degree of a leaf sum, every component of a vector
density and every element's own integral keeps the accuracy of its own terms.

Reference: the recursions of Lemmas 1-4 in numpy's long double (64 or 113
bits), for the first eight leaves.  Tolerance: the library rounds an element's
entry a few times a degree, so 4 (p + 4) units of 2^-53 of the element's largest
entry of the degree, summed over the elements.  The Jacobian, a factor of all
of an element's entries whose own rounding depends on its shape, is the
library's: that of the element alone in a leaf."""
import math

import numpy as np
import pytest
from _helpers import NV, scale_vector

pytestmark = pytest.mark.gpu
KINDS = [("segment", "const"), ("triangle", "const"), ("triangle", "linear"), ("tetra", "const")]
SHAPES = ["heavy core", "light rim", "weights apart", "high degrees"]


@pytest.fixture(scope="module")
def q2x():
    import paper_2107_10942_gb300 as q
    return q


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def leaves(kind, shape, sizes, seed):
    """Elements about the origin of each leaf: vertices per corner, leaf of each, weights."""
    rng = np.random.default_rng(seed)
    n = int(sum(sizes))
    leaf_of = np.repeat(np.arange(len(sizes)), sizes)
    base = rng.uniform(-1, 1, (3, n))
    w = rng.uniform(0.5, 1, n) * rng.choice([-1.0, 1.0], n)
    rim = rng.random(n) < 0.1
    if shape in ("heavy core", "light rim"):
        base[:, ~rim] *= 0.02
        w[rim] *= {"heavy core": 1e-4, "light rim": 1e-9}[shape]
    if shape == "weights apart":
        w *= 10.0 ** rng.uniform(-8, 0, n)
    size = 0.004 if shape != "high degrees" else 0.2
    c = rng.uniform(-3, 3, (3, len(sizes)))
    corners = [c[:, leaf_of] + base + size * rng.standard_normal((3, n)) for _ in range(NV[kind])]
    return corners, leaf_of, w, c


def by_degree(a, p):
    """Per row, the largest magnitude of every degree, (rows, p + 1)."""
    return np.stack([np.abs(a[:, n * n:(n + 1) ** 2]).max(axis=1) for n in range(p + 1)], axis=1)


def entries(kind, corners, c, p, density=None):
    """Per element and packed column, the moments (layers 0 and 1) in long double;
    density: None for one, or the values at the corners."""
    LD, CLD = np.longdouble, np.clongdouble
    x = [k.astype(LD) - c for k in corners]
    e = [corners[k].astype(LD) - corners[0] for k in range(1, len(corners))]
    cross = lambda a, b: np.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])  # noqa: E731
    q = cross(e[0], e[1]) if len(e) > 1 else e[0]
    J = np.abs((q * e[2]).sum(0)) if len(e) > 2 else np.sqrt((q * q).sum(0))
    stencil = [((-v[1] + 1j * v[0]) / 2, (v[1] + 1j * v[0]) / 2, v[2]) for v in x + ([q / J] if len(e) == 2 else [])]
    one = np.ones(J.size, CLD)

    def times(row, k, n):  # the stencil of vertex k on a row of degree n - 1
        xi, eta, z = stencil[k]
        g = lambda m: (row[m] if m >= 0 else (-1) ** m * np.conj(row[-m])) if abs(m) < n else 0  # noqa: E731
        return [xi * g(m - 1) + eta * g(m + 1) - z * g(m) for m in range(n + 1)]

    add = lambda a, b: [u + v for u, v in zip(a, b)]  # noqa: E731
    order = list(range(1, len(x))) + [0]
    if density is None:
        rows, d = [[one] for _ in order], len(order) - 1
    else:
        s, d = [k.astype(LD) for k in density], 3
        rows = [[one], [one], [one * (s[1] + s[2])], [one], [one * (s[0] + s[1] + s[2])]]
    out = [np.zeros((J.size, (p + 1) ** 2), LD) for _ in range(2)]
    for n in range(p + 1):
        last = rows[-1]
        if n and density is None:
            new = []
            for k, row in zip(order, rows):
                new.append(times(row, k, n) if not new else add(times(row, k, n), new[-1]))
            rows = new
        elif n:
            q0 = times(rows[0], 1, n)
            q1 = add(times(rows[1], 2, n), q0)
            E = add(times(rows[2], 2, n), [s[1] * (n + 1) * u + s[2] * v for u, v in zip(q0, q1)])
            i = add(times(rows[3], 0, n), q1)
            rows = [q0, q1, E, i, add(times(rows[4], 0, n), add(E, [s[0] * u for u in i]))]
        for layer, row, f in ((0, rows[-1], n + d), (1, times(last, 3, n) if n and len(x) == 3 else [], n + d - 1)):
            for m, v in enumerate(row):
                v = v * (J / LD(math.factorial(f)))
                out[layer][:, n * n + n + m] = v.real
                if m:
                    out[layer][:, n * n + n - m] = v.imag
    return out


def close_by_degree(got, rows, leaf_of, p):
    s = scale_vector(p, 1.0)
    nl = leaf_of[-1] + 1
    want, size = np.zeros((nl, (p + 1) ** 2), rows.dtype), np.zeros((nl, p + 1))
    np.add.at(want, leaf_of, rows * s)
    np.add.at(size, leaf_of, by_degree(rows * s, p).astype(float))
    err = by_degree(got[:nl] * s - want, p).astype(float)
    bad = err > 4 * (p + 4) * 2.0 ** -53 * size
    assert not bad.any(), (np.argwhere(bad)[:3], (err / np.where(size > 0, size, 1.0)).max(axis=0))


SIZES = [96, 7, 150, 1, 40, 300, 0, 64] * 9  # full tiles, parts of one, several
CHECKED = sum(SIZES[:8])


@pytest.mark.parametrize("kind,density", KINDS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("p", [1, 4, 11, 20])
def test_every_degree_of_a_leaf_sum(q2x, kind, density, shape, p):
    corners, leaf_of, w, c = leaves(kind, shape, SIZES, seed=p)
    n = len(w)
    idx = np.stack([np.arange(n) + k * n for k in range(NV[kind])]).astype(np.int32)
    sigma = np.tile(w, NV[kind]) * np.random.default_rng(p).uniform(0.5, 1, NV[kind] * n) if density == "linear" else w
    off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    plan = q2x.Plan(p, norm="moment")

    a = (dev(np.concatenate(corners, 1)), dev(idx), dev(sigma), dev(off), dev(c))
    if kind == "triangle":
        got = plan.triangles(*a, density=density, single=True, double=True)
    else:
        got = [plan.segments(*a) if kind == "segment" else plan.tetra(*a)]
    plan.sync()
    k = slice(0, CHECKED)
    alone = (*a[:3], dev(np.arange(n + 1)), dev(c[:, leaf_of]))
    alone = (plan.triangles(*alone, density=density)[0] if kind == "triangle" else
             plan.segments(*alone) if kind == "segment" else plan.tetra(*alone)).cpu().numpy()[k, 0]
    values = [sigma[j * n:j * n + CHECKED] for j in range(3)] if density == "linear" else None
    rows = entries(kind, [v[:, k] for v in corners], c[:, leaf_of[k]], p, values)
    factor = (alone / rows[0][:, 0])[:, None]
    for g, r in zip(got, rows):
        close_by_degree(g.cpu().numpy(), r * factor, leaf_of[k], p)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("p", [2, 12, 20])
def test_every_component_of_a_vector_density(q2x, shape, p):
    corners, leaf_of, w, c = leaves("segment", shape, SIZES, seed=p + 40)
    n = len(w)
    rng = np.random.default_rng(p)
    cur = np.stack([w * rng.uniform(0.5, 1, n) * f for f in (1.0, 1e-12, 1e6)])
    cur[1, ::3] = 0.0  # a component that some elements have not
    off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    idx = np.stack([np.arange(n), np.arange(n) + n]).astype(np.int32)
    plan = q2x.Plan(p, norm="moment")
    v = dev(np.concatenate(corners, 1))
    got = plan.segments_vector(v, dev(idx), dev(cur), dev(off), dev(c)).cpu().numpy()
    k = slice(0, CHECKED)
    rows = entries("segment", [x[:, k] for x in corners], c[:, leaf_of[k]], p)[0]
    for j in range(3):
        close_by_degree(got[j], rows * cur[j, k, None], leaf_of[k], p)


@pytest.mark.parametrize("layer", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("high", [1.0, 8.0])
@pytest.mark.parametrize("p", [1, 5, 12, 20])
def test_every_element_of_a_receiver(q2x, p, high, shape, layer):
    """Weights of all degrees alike in the leaf's scale, or growing by `high` a degree."""
    corners, leaf_of, w, c = leaves("triangle", shape, SIZES, seed=p + 80)
    n = len(w)
    idx = np.stack([np.arange(n) + k * n for k in range(3)]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    deg = np.concatenate([np.full(2 * k + 1, float(k)) for k in range(p + 1)])
    wt = np.random.default_rng(p).standard_normal((len(SIZES), (p + 1) ** 2)) * scale_vector(p, 1.0) * high ** deg
    plan = q2x.Plan(p, norm="moment")
    v = dev(np.concatenate(corners, 1))
    got = plan.galerkin_triangles(v, dev(idx), dev(wt), dev(off), dev(c), None, dev(w), layer=layer).cpu().numpy()
    plan.sync()
    k = slice(0, CHECKED)
    rows = entries("triangle", [x[:, k] for x in corners], c[:, leaf_of[k]], p)[layer] * w[k, None]
    wt, s = wt[leaf_of[k]], scale_vector(p, 1.0)
    size = (by_degree(rows * s, p) * by_degree(wt / s, p)).sum(axis=1)
    err = np.abs(got[k] - (rows * wt).sum(axis=1))
    assert np.all(err <= 4 * (p + 4) * 2.0 ** -53 * size), (err / size).max()
