"""Balanced subspace calls (k = n / 2) from the Dicke state whose cost is symmetric (C(z) = C(~z)) run on
half the state; any other cost runs on all of it.  One unit in the last place of one float64 cost
makes a cost asymmetric without moving a result, so both forms run on the same problem.

Tolerances: each form is within 1e-12 (complex128) or 2e-5 (complex64) per amplitude and within
1e-10 max(1, sum|w|) or 1e-4 max(1, |value|) in <C> and gradients, so two forms differ by twice that.
"""
from math import comb

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


@pytest.mark.parametrize("n", [26, 28])
@pytest.mark.parametrize("weights", ["int", "u01"])
@pytest.mark.parametrize("dtype,ta", [("c128", 1e-12), ("c64", 2e-5)])
def test_half_against_whole(n, weights, dtype, ta):
    k, p = n // 2, 2
    e, w, integer = synth.graph("gnp", n, n, weights, prob=0.3)
    g = q.Graph(n, e, w, integer)
    gam, bet = synth.angles(p, n)
    scale = max(1.0, float(np.sum(np.abs(w))))
    states, outs, grads = [], [], []
    for form in ("i32" if integer else "f64", "whole"):
        cv = q.xy_cost_vector(g, k, "f64" if form == "whole" else form)
        if form == "whole":
            r = comb(n, k) // 3
            cv.C[r] = torch.nextafter(cv.C[r], torch.full_like(cv.C[r], 1e300))
        psi, lam = q.xy_new_state(n, k, dtype), q.xy_new_state(n, k, dtype)
        outs.append(q.xy_apply_layers(psi, n, k, cv, gam, bet, expect=True).cpu().numpy())
        states.append(psi.clone())
        grads.append(q.xy_gradient(psi, lam, n, k, cv, gam, bet).cpu().numpy())
        dicke = torch.max(torch.abs(psi - 1.0 / np.sqrt(comb(n, k)))).item()
        assert dicke <= ta  # the adjoint pass undoes every gate, on the whole buffer
    tol = lambda ref: 1e-10 * scale if dtype == "c128" else 1e-4 * np.maximum(1.0, np.abs(ref))  # noqa: E731
    assert torch.max(torch.abs(states[0] - states[1])).item() <= 2 * ta
    assert np.all(np.abs(outs[0] - outs[1]) <= 2 * tol(outs[1]))
    assert np.all(np.abs(grads[0] - grads[1]) <= 2 * tol(grads[1]))
    assert np.all(np.abs(grads[0][:2] - outs[0]) <= 2 * tol(outs[0]))
