"""Two plans in two host threads: the direction kernels of small and large
degree bounds share functions, whose limits on shared memory must not depend
on the call made last."""
import threading

import pytest
from _helpers import random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["triangle", "segment"])
def test_two_plans_in_two_threads(kind):
    import torch

    import paper_2107_10942_gb300 as q2x
    from paper_2107_10942_gb300.q2x import problem_to_device
    made, wrong = [], []
    for p in (20, 2):
        st = torch.cuda.Stream()
        prob = random_problem(kind, [300] * 40, seed=p, p=p)
        d = problem_to_device({k: v for k, v in prob.items() if hasattr(v, "shape")})
        plan = q2x.Plan(p, stream=st)
        call = plan.segments if kind == "segment" else plan.triangles
        out = lambda r: r[0] if isinstance(r, tuple) else r  # noqa: E731
        run = lambda call=call, d=d: out(call(d["vxyz"], d["idx"], d["sigma"], d["leaf_off"], d["leaf_c"]))  # noqa: E731
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            made.append((plan, st, run, run()))
    start = threading.Barrier(2)

    def work(plan, st, run, ref):
        try:
            start.wait(timeout=60)
            with torch.cuda.stream(st):
                for _ in range(6000):
                    got = run()
                plan.sync()
                if not torch.equal(got, ref):
                    wrong.append("bits")
        except Exception as err:  # noqa: BLE001
            wrong.append(repr(err))

    threads = [threading.Thread(target=work, args=m) for m in made]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    assert not wrong, wrong
