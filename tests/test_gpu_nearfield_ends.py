"""The near field exactly at a segment's ends: the potential is infinite,
whatever the signs of the zeros that the offsets' products leave."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_target_at_an_end():
    import torch

    import paper_2107_10942_gb300 as q2x
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    a = np.array([0.5, -0.25, 1.0])
    dirs = [np.array(s) * (3.0, 4.0, 12.0) for s in itertools.product((-1.0, 0.0, 1.0), repeat=3) if any(s)]
    v = np.array([x for d in dirs for x in (a, a + d)])
    n = len(dirs)
    plan = q2x.Plan(2)
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda")
    idx = T(np.arange(2 * n, dtype=np.int32).reshape(n, 2).T)
    for end in (0, 1):
        got = plan.nearfield("segment", T(v.T), idx, T(np.ones(n)), T(v[end::2].T), off, off[:-1].contiguous())
        plan.sync()
        assert torch.isinf(got).all() and (got > 0).all(), (end, got)
