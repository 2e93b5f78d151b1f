"""complex128 gradients with float64 costs at the ends of their range.

A cost entry that is infinite or NaN reaches dE/dgamma, which sums over C, as a non-finite number.

Costs of any scale: with C 2^-k and gamma 2^k the state is the same and dE/dgamma scales by 2^-2k.  The
only rounding that does not scale is lambda's, to 2^-54 per component at 2^12 tiles (less on smaller
ones): psi and lambda meet it once when lambda is formed and once per group and undone mixer, each of
2-norm at most 0.41 x 2^((n + 12)/2 - 54), and it enters dE/dgamma times 2 max |C|.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


def problem(n, scale=1.0):
    e, w, integer = synth.graph("gnp", n, n, "u01", prob=0.3)
    w = np.asarray(w) * scale
    return q.cost_vector(q.Graph(n, e, w, integer), "f64"), float(np.sum(np.abs(w)))


@pytest.mark.parametrize("n", [6, 12, 14, 19, 21, 23])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_costs_show(n, bad):
    cv, _ = problem(n)
    cv.C[(1 << n) // 3] = bad
    psi, lam = q.new_state(n, "c128"), q.new_state(n, "c128")
    out = q.gradient(psi, lam, cv, [0.3, 0.2], [0.4, 0.1]).cpu().numpy()
    assert not np.isfinite(out[0])
    assert not np.any(np.isfinite(out[2:4]))


@pytest.mark.parametrize("n", [6, 12, 14, 19, 21, 23])
@pytest.mark.parametrize("k", [10, 25, -30])
def test_costs_of_any_scale(n, k):
    p = 2
    gam, bet = synth.angles(p, n)
    outs = []
    for f in (1.0, 2.0 ** -k):
        cv, S = problem(n, f)
        psi, lam = q.new_state(n, "c128"), q.new_state(n, "c128")
        outs.append(q.gradient(psi, lam, cv, np.asarray(gam) / f, bet).cpu().numpy())
        if f == 1.0:
            S1 = S
    dg = outs[1][2:2 + p] * 4.0 ** k
    small = 2.0 * S1 * (1 + 6 * p) * 0.41 * 2.0 ** ((n + 12) / 2 - 54) * 2.0 ** max(k, 0)
    assert np.all(np.abs(dg - outs[0][2:2 + p]) <= 1e-10 * S1 * S1 + small)
