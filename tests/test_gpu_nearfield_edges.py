"""The near field's two forms of an edge's logarithm (csrc/q2x_nearfield.cu)
about the distance where one takes over, from close by to far away, against
the closed form in extended precision.

Tolerance: offsets, heights and distances carry a few roundings of 1.1e-16 of
the distance R to the triangle, logarithms and arctangents under one unit of
their own: forty roundings, 4.4e-15, of the sum of R log and |h solid| would
be a bad case; 1e-14."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LD = np.longdouble


def single_layer(X, r):
    """(int 1/|r - y| dS, the size of its terms) over the triangle X in extended precision."""
    X, r = [x.astype(LD) for x in X], r.astype(LD)
    e = [X[(i + 1) % 3] - X[i] for i in range(3)]
    nr = np.cross(e[0], -e[2])
    J = np.sqrt(nr @ nr)
    n = nr / J
    h = (r - X[0]) @ n
    d = [x - r for x in X]
    R = [np.sqrt(v @ v) for v in d]
    S, size = LD(0), LD(0)
    for i in range(3):
        L = np.sqrt(e[i] @ e[i])
        t = d[i] @ np.cross(e[i] / L, n)
        Sg = R[i] + R[(i + 1) % 3]
        log = np.log1p(2 * L / (Sg - L))
        S += t * log
        size += max(R) * log
    den = R[0] * R[1] * R[2] + (d[0] @ d[1]) * R[2] + (d[0] @ d[2]) * R[1] + (d[1] @ d[2]) * R[0]
    solid = 2 * np.arctan2(J * abs(h), den)
    return S - abs(h) * solid, size + abs(h) * solid


@pytest.mark.parametrize("unit", [1.0, 1e-9, 1e12])
def test_edge_forms(unit):
    import torch

    import paper_2107_10942_gb300 as q2x
    rng = np.random.default_rng(4)
    X = [np.array(v) * unit for v in ([0.1, 0.2, -0.1], [1.3, 0.1, 0.2], [0.4, 0.9, 0.5])]
    tgt = []
    for i in range(3):
        a, b = X[i], X[(i + 1) % 3]
        L = np.linalg.norm(b - a)
        l = (b - a) / L
        for x in (1.02, 1.2, 1.4, 1.45, 1.5, 1.55, 1.62, 1.7, 2.0, 3.0, 10.0, 1e3):
            for _ in range(4):
                v = rng.standard_normal(3)
                v -= (v @ l) * l
                tgt.append((a + b) / 2 + v / np.linalg.norm(v) * (L / 2) * np.sqrt(x * x - 1))
    tgt = np.array(tgt)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    plan = q2x.Plan(2)
    got = plan.nearfield("triangle", T(np.array(X).T), T(np.array([[0], [1], [2]], dtype=np.int32)),
                         T(np.ones(1)), T(tgt.T)).cpu().numpy()
    assert plan.device_errors() == 0
    for k, r in enumerate(tgt):
        want, size = single_layer(X, r)
        assert abs(got[k] * 4 * np.pi - float(want)) <= 1e-14 * float(size), (k, got[k], want)
