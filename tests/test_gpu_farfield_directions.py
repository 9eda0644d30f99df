"""The direction path of the far-field evaluation (calls with many targets)
against the general FP64 path (the same targets in shorter calls):
degrees, norms, target lists over several expansions, distances from the
nearest target to 10^4 times it, zero monopoles, targets at a centre, bad
indices, accumulation.

Tolerance: both paths round each degree's term to some (p + 1) units of 2^-53
of its bound sum_m |F_n^m| sqrt((n+m)! (n-m)!) / r^(n+1) (times (n + 1) / r for
the curl); p <= 20 and at most eight expansions keep that below 1e-13 of the
bounds' sum."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q2x():
    import paper_2107_10942_gb300 as q
    return q


def expansions(rng, n_exp, p, rho, comps=1):
    out = rng.standard_normal((comps, n_exp, (p + 1) ** 2))
    for n in range(p + 1):
        for m in range(-n, n + 1):
            out[..., n * n + n + m] *= rho ** n / math.sqrt(math.factorial(n + abs(m)) * math.factorial(n - abs(m)))
    return out


def bound(coef, c, x, p, norm, lists, off, curl):
    """Per target the sum over its list of the degrees' bounds."""
    f = np.concatenate([[math.sqrt(math.factorial(n + abs(m)) * math.factorial(n - abs(m))) for m in range(-n, n + 1)]
                        for n in range(p + 1)])
    s = np.stack([np.abs(coef * f)[..., n * n:(n + 1) ** 2].sum(-1).max(0) for n in range(p + 1)])  # (p+1, n_exp)
    out, lists = np.zeros(x.shape[1]), lists.reshape(x.shape[1], -1)
    for i in range(lists.shape[1]):
        e = lists[:, i]
        r = np.linalg.norm(x - c[:, e], axis=0)
        r[r == 0] = np.inf
        for n in range(p + 1):
            out += s[n, e] * ((n + 1) / r if curl else 1.0) / r ** (n + 1)
    return out


@pytest.mark.parametrize("p,norm,n_exp,k", [(2, "coeff", 1, 1), (3, "moment", 3, 2), (7, "coeff", 40, 3),
                                           (12, "coeff", 1, 1), (12, "moment", 8, 8), (16, "coeff", 5, 2),
                                           (20, "moment", 1, 1)])
@pytest.mark.parametrize("curl", [False, True])
def test_against_general_path(q2x, p, norm, n_exp, k, curl):
    import torch
    if curl and norm == "moment":
        norm = "coeff"
    rng = np.random.default_rng(p + n_exp)
    T = (180000 if curl else 3000000) * 2 // ((p + 1) * (p + 2)) + 137  # just past the line of the dispatch
    coef = expansions(rng, n_exp, p, 0.5, 3 if curl else 1)
    coef[:, n_exp // 2, 0] = 0.0  # no monopole
    c = rng.uniform(-0.3, 0.3, (3, n_exp))
    x = rng.standard_normal((3, T))
    x *= rng.uniform(1.6, 3.0, T) / np.linalg.norm(x, axis=0)
    x[:, 100:160] *= 10.0 ** rng.uniform(0.5, 4, 60)  # some far beyond the others
    off = np.arange(T + 1, dtype=np.int64) * k
    lists = rng.integers(0, n_exp, T * k)
    x[:, 7] = c[:, lists[7 * k]]  # at a centre
    plan = q2x.Plan(p, norm=norm)
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (coef if curl else coef[0], c)]
    f = plan.evaluate_curl if curl else plan.evaluate
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = f(d[0], d[1], dev(x), dev(off), dev(lists)).cpu().numpy()
    parts = []
    for a, b in ((0, T // 2), (T // 2, T)):
        parts.append(f(d[0], d[1], dev(x[:, a:b]), dev(off[a:b + 1] - off[a]), dev(lists[a * k:b * k])).cpu().numpy())
    ref = np.concatenate(parts, axis=-1)
    plan.sync()
    tol = 1e-13 * bound(coef, c, x, p, norm, lists, off, curl) / (1.0 if norm == "coeff" else 4 * math.pi)
    assert np.all(np.abs(got - ref) <= tol)
    base = torch.rand(*got.shape, dtype=torch.float64, device="cuda")
    acc = base.clone()
    f(d[0], d[1], dev(x), dev(off), dev(lists), out=acc, accumulate=True)
    assert torch.equal(acc.cpu(), base.cpu() + torch.from_numpy(got))


def test_input_errors_and_infinities(q2x):
    """A bad expansion index contributes zero and is reported; an infinite
    coefficient gives what the general path gives."""
    import torch
    rng = np.random.default_rng(5)
    p, T = 9, 60000
    plan = q2x.Plan(p)
    coef = torch.from_numpy(expansions(rng, 2, p, 0.5)[0]).cuda()
    c = torch.zeros(3, 2, dtype=torch.float64, device="cuda")
    x = torch.from_numpy(rng.uniform(1.0, 2.0, (3, T))).cuda()
    off = torch.arange(T + 1, dtype=torch.int64, device="cuda")
    idx = torch.zeros(T, dtype=torch.int64, device="cuda")
    good = plan.evaluate(coef, c, x, off, idx)
    idx[5], idx[6] = 2, -1
    out = plan.evaluate(coef, c, x, off, idx)
    assert plan.device_errors() & 1
    assert out[5] == 0 and out[6] == 0 and torch.equal(out[7:], good[7:])
    idx[5] = idx[6] = 0
    coef[0, 3] = float("inf")
    got = plan.evaluate(coef, c, x, off, idx)
    ref = torch.cat([plan.evaluate(coef, c, x[:, a:a + T // 3].contiguous(), off[:T // 3 + 1], idx[:T // 3]) for a in range(0, T, T // 3)])
    assert torch.equal(torch.isnan(got), torch.isnan(ref)) and torch.equal(torch.isinf(got), torch.isinf(ref))
