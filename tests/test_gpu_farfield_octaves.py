"""The direction path of the far field where an expansion's targets lie in many
octaves of distance: many in two of them, few in others (a target inside the
expansion's sphere, one a power of two to the sixteenth farther), against the
general path (the same targets in shorter calls), with the tolerance of
test_gpu_farfield_directions.py."""
import math

import numpy as np
import pytest
from test_gpu_farfield_directions import bound, expansions

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n_exp,k", [(2, 1, 1), (9, 6, 3), (12, 1, 1), (20, 2, 1)])
@pytest.mark.parametrize("curl", [False, True])
def test_targets_in_many_octaves(p, n_exp, k, curl):
    import torch

    import paper_2107_10942_gb300 as q2x
    rng = np.random.default_rng(p + n_exp)
    T = (180000 if curl else 3000000) * 2 // ((p + 1) * (p + 2)) + 61  # past the line of the dispatch
    coef = expansions(rng, n_exp, p, 0.4, 3 if curl else 1)
    c = rng.uniform(-0.1, 0.1, (3, n_exp))
    x = rng.standard_normal((3, T))
    x *= rng.uniform(1.1, 1.9, T) / np.linalg.norm(x, axis=0)
    x[:, ::3] *= 2.0
    for i, f in ((11, 0.01), (200, 0.25), (201, 0.251), (333, 2.0 ** 16), (334, 2.0 ** 17), (400, 2.0 ** -16), (401, 1e6)):
        x[:, i] *= f
    off = np.arange(T + 1, dtype=np.int64) * k
    lists = rng.integers(0, n_exp, T * k)
    plan = q2x.Plan(p)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    f = plan.evaluate_curl if curl else plan.evaluate
    d = [dev(coef if curl else coef[0]), dev(c)]
    run = lambda a, b: f(*d, dev(x[:, a:b]), dev(off[a:b + 1] - off[a]), dev(lists[a * k:b * k])).cpu().numpy()  # noqa: E731
    launches = plan.launch_count()
    got = run(0, T)
    assert plan.launch_count() - launches == 3  # the direction path
    assert np.array_equal(got, run(0, T))
    ref = np.concatenate([run(0, T // 2), run(T // 2, T)], axis=-1)
    plan.sync()
    assert np.all(np.abs(got - ref) <= 1e-13 * bound(coef, c, x, p, "coeff", lists, off, curl))
