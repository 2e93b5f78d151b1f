"""complex128 gradients with float64 costs whose largest entry is a power of two, the end of the range of
the fixed-point cost: the same costs in int32 give the same gradient.  Each is within 1e-10 of the exact
one in units of max(1, sum|w|), so the two differ by at most twice that.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


@pytest.mark.parametrize("n,m", [(6, 4), (11, 8), (14, 8), (18, 16), (19, 16), (20, 16), (22, 16), (24, 16)])
@pytest.mark.parametrize("weight", [1.0, 64.0])
def test_power_of_two_maximum(n, m, weight):
    e = np.array([[i, i + 1] for i in range(m)], dtype=np.int32)  # a path: every edge can be cut
    g = q.Graph(n, e, np.full(m, weight), True)
    gam, bet = synth.angles(2, n)
    gam = np.asarray(gam) / weight
    out = []
    for dtype in ("i32", "f64"):
        cv = q.cost_vector(g, dtype)
        assert cv.C.max().item() == m * weight
        psi, lam = q.new_state(n, "c128"), q.new_state(n, "c128")
        out.append(q.gradient(psi, lam, cv, gam, bet).cpu().numpy())
    scale = m * weight
    tol = 2e-10 * np.array([scale, 1.0] + [scale * scale] * 2 + [scale] * 2)
    assert np.all(np.abs(out[0] - out[1]) <= tol)
