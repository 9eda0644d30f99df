"""The FP32 adjoint kernel where leaves of several degrees meet in a warp and
at the edges of warps, against the FP64 kernel of the same library.

Tolerance: p stencil steps of three FMAs each carry 3 p 2^-24 <= 3.6e-6 of the
magnitudes at p = 20; (p + 1)^2 columns with random weights sum to about 1/21
of their magnitudes there: 1e-4 of the largest component."""
import numpy as np
import pytest
from _helpers import random_problem

pytestmark = pytest.mark.gpu


def grads(q2x, prob, p, G, precision, rho=True):
    import torch
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    plan = q2x.Plan(p, precision=precision)
    gv, gs = plan.triangles_single_vjp(T(prob["vxyz"]), T(prob["idx"]), T(prob["sigma"]), T(prob["leaf_off"]),
                                       T(prob["leaf_c"]), T(G), T(prob["leaf_rho"]) if rho else None,
                                       T(prob["leaf_p"]))
    errors = plan.device_errors()
    return gv.cpu().numpy(), gs.cpu().numpy(), errors


@pytest.mark.parametrize("p", [0, 1, 4, 7, 8, 11, 12, 13, 16, 19, 20])
def test_mixed_degrees(q2x, p):
    sizes = [1, 0, 31, 32, 33, 0, 0, 2, 1, 1, 3, 60, 64, 95, 5, 0, 17]
    prob = random_problem("triangle", sizes, seed=p, p=p)
    rng = np.random.default_rng(p)
    n = np.array([k for k in range(p + 1) for _ in range(2 * k + 1)])
    fact = np.cumprod(np.concatenate([[1.0], np.arange(1.0, p + 1)]))
    G = rng.standard_normal((len(sizes), (p + 1) ** 2)) * (fact[n] / prob["leaf_rho"][:, None] ** n)
    prob["leaf_p"] = rng.integers(0, p + 1, len(sizes)).astype(np.int32)
    prob["leaf_p"][2] = p
    for bad in (False, True):
        if bad:
            prob["leaf_p"][[4, 9]] = [p + 1, -1]  # their elements: error bit and zeros
        v64, s64, e64 = grads(q2x, prob, p, G, "fp64")
        v32, s32, e32 = grads(q2x, prob, p, G, "fp32")
        assert e32 == e64 == (4 if bad else 0)
        assert np.max(np.abs(v32 - v64)) <= 1e-4 * np.max(np.abs(v64))
        assert np.max(np.abs(s32 - s64)) <= 1e-4 * np.max(np.abs(s64))
        if bad:
            off = prob["leaf_off"]
            assert not s32[off[4]:off[5]].any() and not s32[off[9]:off[10]].any()


def test_low_degree_beside_high_degree(q2x):
    """Unscaled leaves: the powers of a far element overflow FP32 beyond its own
    degree, which only its neighbour's degree reaches."""
    p = 20
    prob = random_problem("triangle", [4, 4], seed=3, p=p)
    far = np.unique(prob["idx"][:, :4])
    assert not np.intersect1d(far, prob["idx"][:, 4:]).size
    prob["vxyz"][:, far] *= 1e6
    prob["leaf_c"][:, 0] *= 1e6
    prob["leaf_p"] = np.array([1, p], dtype=np.int32)
    G = np.random.default_rng(1).standard_normal((2, (p + 1) ** 2))
    v64, s64, _ = grads(q2x, prob, p, G, "fp64", rho=False)
    v32, s32, _ = grads(q2x, prob, p, G, "fp32", rho=False)
    near = np.unique(prob["idx"][:, 4:])
    for sel, el in ((far, slice(0, 4)), (near, slice(4, 8))):
        assert np.max(np.abs(v32 - v64)[:, sel]) <= 1e-4 * np.max(np.abs(v64[:, sel]))
        assert np.max(np.abs(s32 - s64)[el]) <= 1e-4 * np.max(np.abs(s64[el]))


@pytest.fixture(scope="module")
def q2x():
    import paper_2107_10942_gb300 as q
    return q
