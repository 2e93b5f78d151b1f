"""The batch's cost tables at the sizes where they can go wrong: fewer than 16 entries, one side of
each six-bit half and of the 2^12 block; negative and float weights.  Each row's <C> and gradient
against the oracle within 1e-10 max(1, sum|w|)."""
import numpy as np
import pytest

import synth
from oracle import qaoa

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


@pytest.mark.parametrize("weights", ["int", "u01"])
def test_batch_costs(weights):
    p, graphs, ang, want, tol = 2, [], [], [], []
    for n in (2, 3, 4, 5, 6, 7, 11, 12, 13, 14):
        for lo in ((-5, 1) if weights == "int" else (0,)):
            e, w, integer = synth.graph("gnp", n, n, weights, prob=0.8, lo=lo, hi=9)
            gam, bet = synth.angles(p, n)
            C = qaoa.cut_values(n, e, w, integer=integer)
            E, dg, db, _ = qaoa.adjoint_gradient(n, C, gam, bet)
            graphs.append(q.Graph(n, e, w, integer))
            ang.append(np.concatenate([gam, bet]))
            want.append(np.concatenate([[E, 1.0], dg, db]))
            tol.append(1e-10 * max(1.0, float(np.sum(np.abs(w)))))
    got = q.batch_gradient(graphs, np.stack(ang), "c128").cpu().numpy()
    assert np.all(np.abs(got - np.stack(want)) <= np.array(tol)[:, None])
