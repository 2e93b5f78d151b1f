"""Batched gradients with float weights at the bottom of float64's range: costs may be subnormal.  Without a
cost unitary (gamma = 0) the state stays |+> up to a phase, whose <C> is sum w / 2: within 1e-10 sum|w|.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


@pytest.mark.parametrize("scale", [1e-280, 1e-300, 1e-305])
def test_subnormal_costs(scale):
    graphs, want = [], []
    for n in (3, 5, 12, 13, 20):
        e = np.array([[i, i + 1] for i in range(n - 1)], dtype=np.int32)
        w = scale * np.array([1e-5 if i == 1 else 1.0 for i in range(n - 1)])  # a cost of one light edge
        graphs.append(q.Graph(n, e, w, False))
        want.append(float(np.sum(w)) / 2)
    got = q.batch_gradient(graphs, np.tile([0.0, 0.3], (len(graphs), 1)), "c128").cpu().numpy()
    assert np.all(np.abs(got[:, 0] - want) <= 2e-10 * np.array(want))
