"""A plan and a batch that go away while another plan's calls are captured
(the garbage collector may choose that moment): the capture stays valid."""
import numpy as np
import pytest
from _helpers import random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["plan", "batch"])
def test_released_while_another_is_captured(what):
    import torch

    import paper_2107_10942_gb300 as q2x
    from paper_2107_10942_gb300.q2x import Batch, problem_to_device
    prob = random_problem("triangle", [30, 200], seed=1, p=4)
    d = problem_to_device({k: v for k, v in prob.items() if hasattr(v, "shape")})
    args = (d["vxyz"], d["idx"], d["sigma"], d["leaf_off"], d["leaf_c"])
    old = q2x.Plan(4)
    old.triangles(*args)
    batch = None
    if what == "batch":
        tri = dict(vxyz=d["vxyz"], idx=d["idx"], sigma=d["sigma"], leaf_off=d["leaf_off"])
        batch = Batch(old, d["leaf_c"], triangles=tri)
        batch.run()
    plan = q2x.Plan(4)
    ref = plan.triangles(*args)[0].clone()
    out = torch.zeros_like(ref)
    torch.cuda.synchronize()
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    plan.set_stream(side)
    with torch.cuda.graph(graph, stream=side):
        plan.triangles(*args, coef_single=out)
        if batch is not None:
            batch.close()
        old.close()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    assert np.isfinite(out.cpu().numpy()).all()
