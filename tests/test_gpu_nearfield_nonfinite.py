"""The near field at targets that are not numbers: the result says so."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

X = np.array([[0.1, 0.2, -0.1], [1.3, 0.1, 0.2], [0.4, 0.9, 0.5], [0.3, 0.4, 1.4]])


@pytest.mark.parametrize("kind,layer", [("segment", 0), ("triangle", 0), ("triangle", 1), ("tetra", 0)])
def test_nan_target_stays_nan(kind, layer):
    import torch

    import paper_2107_10942_gb300 as q2x
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    k = {"segment": 2, "triangle": 3, "tetra": 4}[kind]
    tgt = np.full((3, 5), 0.7)
    for d in range(3):
        tgt[d, d] = np.nan
    tgt[:, 3] = np.nan
    plan = q2x.Plan(2)
    got = plan.nearfield(kind, T(X.T), T(np.arange(k, dtype=np.int32)[:, None]), T(np.ones(1)), T(tgt),
                         layer=layer).cpu().numpy()
    assert np.isnan(got[:4]).all(), got
    assert np.isfinite(got[4])


def test_nan_vertex_gives_zero():
    # a face without an area contributes nothing
    import torch

    import paper_2107_10942_gb300 as q2x
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    bad = X.copy()
    bad[0, 1] = np.nan
    plan = q2x.Plan(2)
    tgt = T(np.full((3, 1), 0.7))
    for layer in (0, 1):
        got = plan.nearfield("triangle", T(bad.T), T(np.arange(3, dtype=np.int32)[:, None]), T(np.ones(1)), tgt,
                             layer=layer)
        assert got.item() == 0.0
