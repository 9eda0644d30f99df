"""q2x_leaf_reduce: rows summed in element order (the same bits as a loop) for
leaves about the eight rows of a step and column counts about a warp, and bad
offsets reported whichever of them is bad."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [0, 4, 5, 20])
def test_sums_and_offset_check(p):
    import torch

    import paper_2107_10942_gb300 as q2x
    rng = np.random.default_rng(p)
    sizes = [0, 1, 7, 8, 9, 0, 16, 17, 300, 0]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    elem = rng.standard_normal((off[-1], (p + 1) ** 2)) * 10.0 ** rng.uniform(-5, 5, (off[-1], 1))
    plan = q2x.Plan(p)
    e = torch.from_numpy(elem).cuda()
    got = plan.leaf_reduce(e, p, torch.from_numpy(off).cuda())
    acc = plan.leaf_reduce(e, p, torch.from_numpy(off).cuda(), coef=got.clone(), accumulate=True)
    assert plan.device_errors() == 0
    for k in range(len(sizes)):
        want = np.zeros(elem.shape[1])
        for r in elem[off[k]:off[k + 1]]:
            want = want + r
        assert np.array_equal(got[k].cpu().numpy(), want)
    assert torch.equal(acc, 2 * got)
    for at, v in ((0, 1), (len(sizes), off[-1] - 1), (len(sizes), off[-1] + 1), (5, off[-1] + 5), (5, -1), (3, off[5])):
        bad = off.copy()
        bad[at] = v
        plan.leaf_reduce(e, p, torch.from_numpy(bad).cuda())
        assert plan.device_errors() & 8
