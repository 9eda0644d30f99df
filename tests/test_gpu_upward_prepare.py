"""Preparing an upward pass: no shift rows for levels that are translated by
octants, rows where leaves are centred elsewhere in their boxes, and rows of
every level for a caller that asks for them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off_centre", [False, True])
def test_rows_only_where_a_pass_takes_them(off_centre):
    import torch

    import paper_2107_10942_gb300 as q2x
    from paper_2107_10942_gb300.upward import Upward
    p, depth, lo, size = 5, 4, -1.1, 2.3
    rng = np.random.default_rng(3)
    ijk = np.unique(rng.integers(0, 1 << depth, (200, 3)), axis=0)
    h = size / (2 << depth)
    leaf_c = lo + (ijk.T + 0.5) * (2 * h)
    if off_centre:
        leaf_c = leaf_c + 0.1 * h * rng.uniform(-1, 1, leaf_c.shape)
    plan = q2x.Plan(p)
    before = plan.launch_count()
    up = Upward(plan, leaf_c, lo, size, depth, device="cuda")
    assert plan.launch_count() - before == int(off_centre)  # the rows of the deepest level alone
    coef = torch.from_numpy(rng.standard_normal((len(ijk), (p + 1) ** 2))).cuda()
    got = [x.clone() for x in up.run(coef)]
    for a, b in zip(got, up.run(coef, precomputed_shifts=False)):
        assert float((a - b).abs().max()) <= 1e-12 * float(b.abs().max())
    assert len(up.rt) == depth and all(rt.shape[1] == (p + 1) ** 2 for rt, _ in up.rt)
