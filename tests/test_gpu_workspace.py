"""The memory behind captured calls and q2x_reserve: what a captured graph
uses stays its own when later calls on the plan need more."""
import numpy as np
import pytest

from _helpers import random_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q2x():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_10942_gb300 import build
    build.build()
    import paper_2107_10942_gb300 as q
    return q


def _targets(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    d = torch.randn(3, n, dtype=torch.float64, device="cuda", generator=g)
    return (d / d.norm(dim=0) * (2.0 + torch.rand(n, dtype=torch.float64, device="cuda", generator=g))).contiguous()


def _lists(n, n_exp=1):
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda")
    return off, off[:-1] % n_exp


def _far(n_exp, p, seed, comps=None):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (n_exp, (p + 1) ** 2) if comps is None else (comps, n_exp, (p + 1) ** 2)
    coef = torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
    for n in range(1, p + 1):
        coef[..., n * n:(n + 1) ** 2] *= 0.5 ** n / float(np.prod(np.arange(1.0, n + 1)))
    return coef, 0.1 * torch.rand(3, n_exp, dtype=torch.float64, device="cuda", generator=g)


@pytest.mark.parametrize("curl", [False, True])
def test_captured_far_field_keeps_its_scratch(q2x, curl):
    p, n = 6, 120_000
    plan = q2x.Plan(p)
    f = plan.evaluate_curl if curl else plan.evaluate
    coef, c = _far(1, p, 1, 3 if curl else None)
    tgt = _targets(n, 2)
    off, idx = _lists(n)
    out = torch.empty((3, n) if curl else n, dtype=torch.float64, device="cuda")
    graph = plan.capture(lambda: f(coef, c, tgt, off, idx, out=out))
    ref = out.clone()
    held = plan.workspace_bytes()
    # larger calls of the same kind and of others grow the plan's buffers
    coef2, c2 = _far(4000, p, 3, 3 if curl else None)
    n2 = 120_000
    f(coef2, c2, _targets(n2, 4), *_lists(n2, 4000))
    plan.reserve(2_000_000, 1000)
    torch.empty(64 << 20, dtype=torch.uint8, device="cuda").fill_(0xff)
    assert plan.workspace_bytes() > held
    out.zero_()
    graph.replay()
    plan.sync()
    assert torch.equal(out, ref)


def test_captured_far_field_beside_the_plans_calls(q2x):
    """A replay on one stream and eager calls on another share no scratch."""
    p, n = 8, 1 << 17
    plan = q2x.Plan(p)
    coef, c = _far(1, p, 5)
    tgt = _targets(n, 6)
    off, idx = _lists(n)
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    graph = plan.capture(lambda: plan.evaluate(coef, c, tgt, off, idx, out=out))
    coef_b, c_b = _far(1, p, 7)
    ref = out.clone()
    ref_b = plan.evaluate(coef_b, c_b, tgt, off, idx)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(30):
        with torch.cuda.stream(side):
            graph.replay()
        got_b = plan.evaluate(coef_b, c_b, tgt, off, idx)
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and torch.equal(got_b, ref_b)


def test_far_field_scratch_follows_the_stream(q2x):
    p, n = 8, 1 << 17
    plan = q2x.Plan(p)
    probs = [_far(1, p, 10 + i) for i in range(4)]
    tgt = _targets(n, 8)
    off, idx = _lists(n)
    ref = [plan.evaluate(a, b, tgt, off, idx) for a, b in probs]
    home = torch.cuda.current_stream()
    streams = [torch.cuda.Stream() for _ in probs]
    torch.cuda.synchronize()
    outs = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in probs]
    for _ in range(10):
        for (a, b), st, o in zip(probs, streams, outs):
            plan.set_stream(st)
            plan.evaluate(a, b, tgt, off, idx, out=o)
    plan.set_stream(home)
    torch.cuda.synchronize()
    for o, r in zip(outs, ref):
        assert torch.equal(o, r)


def test_graph_scratch_is_given_back(q2x):
    p, n = 6, 120_000
    plan = q2x.Plan(p)
    coef, c = _far(1, p, 1)
    tgt = _targets(n, 2)
    off, idx = _lists(n)
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    sizes = []
    for _ in range(6):
        graph = plan.capture(lambda: plan.evaluate(coef, c, tgt, off, idx, out=out))
        graph.replay()
        torch.cuda.synchronize()
        graph.graph.reset()
        del graph
        sizes.append(plan.workspace_bytes())
    assert sizes[-1] <= sizes[0] + 2 * (sizes[1] - sizes[0]) + (1 << 20)


def test_captured_elements_survive_growth(q2x):
    from paper_2107_10942_gb300.q2x import problem_to_device
    prob = random_problem("triangle", [40, 0, 700, 3, 130], seed=31, p=8)
    d = problem_to_device({k: v for k, v in prob.items() if hasattr(v, "shape")})
    plan = q2x.Plan(8)
    out = torch.empty((prob["leaf_c"].shape[1], 81), dtype=torch.float64, device="cuda")

    def step():
        plan.triangles(d["vxyz"], d["idx"], d["sigma"], d["leaf_off"], d["leaf_c"], coef_single=out)

    graph = plan.capture(step)
    ref = out.clone()
    held = plan.workspace_bytes()
    plan.reserve(1_000_000, 1000)
    assert plan.workspace_bytes() > held
    junk = torch.empty(held, dtype=torch.uint8, device="cuda").fill_(0xff)
    out.zero_()
    graph.replay()
    plan.sync()
    assert torch.equal(out, ref)
    del junk


@pytest.mark.parametrize("p,n_res,l_res,calls", [(20, 433, 64, [(311, 64), (433, 1), (152, 64)]),
                                                (12, 9000, 300, [(9000, 300), (4000, 300), (1300, 2), (310, 300)])])
def test_reserve_covers_smaller_calls(q2x, p, n_res, l_res, calls):
    # smaller calls may take smaller tiles and so more of them
    from paper_2107_10942_gb300.q2x import problem_to_device
    plan = q2x.Plan(p)
    plan.reserve(n_res, l_res)
    held = plan.workspace_bytes()
    for n, nl in calls:
        sizes = [n // nl + (1 if k < n % nl else 0) for k in range(nl)]
        prob = random_problem("triangle", sizes, seed=n, p=p)
        d = problem_to_device({k: v for k, v in prob.items() if hasattr(v, "shape")})
        plan.triangles(d["vxyz"], d["idx"], d["sigma"], d["leaf_off"], d["leaf_c"], single=True, double=True)
        plan.triangles(d["vxyz"], d["idx"], d["sigma"], d["leaf_off"], d["leaf_c"])
        plan.sync()
        assert plan.workspace_bytes() == held, (n, nl)
