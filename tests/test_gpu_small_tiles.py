"""complex128 calls around the sizes of the 512-amplitude tiles (one tile, two groups, the last n on
them and the first n past them) against the oracle.  Tolerances: <C> and gradients within
1e-10 max(1, sum|w|), the state within 1e-11 in 2-norm."""
import numpy as np
import pytest

import synth
from oracle import qaoa

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


@pytest.mark.parametrize("n", [2, 8, 9, 10, 11, 12, 13, 18, 19])
@pytest.mark.parametrize("weights", ["int", "u01"])
def test_small_tiles(n, weights):
    e, w, integer = synth.graph("gnp", n, n, weights, prob=0.5)
    C = qaoa.cut_values(n, e, w, integer=integer).astype(np.float64)
    cv = q.cost_vector(q.Graph(n, e, w, integer), "i32" if integer else "f64")
    gam, bet = synth.angles(3, n)
    tol = 1e-10 * max(1.0, float(np.sum(np.abs(w))))
    E, dg, db, _ = qaoa.adjoint_gradient(n, C, gam, bet)
    psi, lam = q.new_state(n, "c128"), q.new_state(n, "c128")
    got = q.gradient(psi, lam, cv, gam, bet).cpu().numpy()
    assert np.all(np.abs(got - np.concatenate([[E, 1.0], dg, db])) <= tol)
    out = q.apply_layers(psi, cv, gam, bet, expect=True).cpu().numpy()
    assert np.all(np.abs(out - [E, 1.0]) <= tol)
    assert np.linalg.norm(psi.cpu().numpy() - qaoa.qaoa_state(n, C, gam, bet)) <= 1e-11
