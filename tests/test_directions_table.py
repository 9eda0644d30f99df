"""The direction tables (gen_directions.py) on the CPU: the vectors are null and
of unit parts, and the left inverses recover random scaled values from their
samples."""
import numpy as np
import pytest

from paper_2107_10942_gb300 import gen_directions as G


def as_float(v):
    return v / (1 << G.FRAC)


@pytest.mark.parametrize("p", [0, 1, 2, 7, 12, 20])
def test_null_vectors_and_left_inverse(p):
    vec, rows = G.samples(p)
    for a in vec:
        a = np.array([complex(as_float(r), as_float(i)) for r, i in a])
        # |Re a| = |Im a| = 1 and a.a = 0, from points rounded to 2^-20 in exact arithmetic
        assert abs(np.sum(a * a)) < 1e-15 and abs(np.linalg.norm(a.real) - 1) < 1e-15
    rng = np.random.default_rng(p)
    for n in range(p + 1):
        A = np.array(rows[n], dtype=object)
        sv = np.linalg.svd((A / G.ONE).astype(float), compute_uv=False)
        assert sv[-1] > 0.7
        X = G.left_inverse(rows[n])
        eye = X.dot(A)
        for i in range(2 * n + 1):
            for j in range(2 * n + 1):
                assert abs((int(eye[i, j]) >> G.FRAC) - (G.ONE if i == j else 0)) < G.ONE >> 90
        # a random row through the rounded table: samples, then the table's halves
        N = rng.standard_normal(2 * n + 1)
        S = (A / G.ONE).astype(float) @ N
        h = np.array([[G.split(int(v), 30, 28) for v in r] for r in X])
        T = h[..., 0] * 2.0 ** -30 + h[..., 1] * 2.0 ** -58
        assert np.max(np.abs(T @ S - N)) < 1e-13 * np.max(np.abs(N))


@pytest.mark.parametrize("v", [0, 1, -1, 3, (1 << G.FRAC) - (1 << (G.FRAC - 31)), (1 << (G.FRAC - 31)) - (1 << G.FRAC), (1 << (G.FRAC - 31)) * 12345 + 99])
def test_split_is_exact_to_its_bits(v):
    h, l = G.split(v, 31, 31)
    got = ((h << 31) + l) << (G.FRAC - 62)
    assert abs(got - v) <= 1 << (G.FRAC - 63)
