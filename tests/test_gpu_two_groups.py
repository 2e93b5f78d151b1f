"""Gradients whose second group carries no or one low bit (n = 23, 24 complex128, 25, 26
complex64): their cost tiles are read in runs below 16 bytes.  Against the p = 1 closed form, and
(p = 2) one batched graph against the one-graph call."""
import numpy as np
import pytest

import synth
from oracle import closed_form

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dtype", [(23, "c128"), (24, "c128"), (25, "c64"), (26, "c64")])
@pytest.mark.parametrize("weights", ["int", "u01"])
def test_short_runs(n, dtype, weights):
    import torch
    import paper_2407_13012_gb300 as q
    e, w, integer = synth.graph("gnp", n, n, weights, prob=0.2)
    gam, bet = synth.angles(2, n)
    g = q.Graph(n, e, w, integer)
    cv = q.cost_vector(g, "i32" if integer else "f64")
    psi, lam = q.new_state(n, dtype), q.new_state(n, dtype)
    out = q.gradient(psi, lam, cv, gam[:1], bet[:1]).cpu().numpy()
    E = closed_form.expectation_p1(n, e, w, gam[0], bet[0])
    ref = np.array([E, 1.0, *closed_form.gradient_p1_exact(n, e, w, gam[0], bet[0])])
    tol = 1e-10 * max(1.0, np.sum(np.abs(w))) if dtype == "c128" else 1e-4 * np.maximum(1.0, np.abs(ref))
    assert np.all(np.abs(out - ref) <= tol), (out, ref)
    one = q.gradient(psi, lam, cv, gam, bet).cpu().numpy()
    del psi, lam, cv
    torch.cuda.empty_cache()
    row = q.batch_gradient([g], np.concatenate([gam, bet])[None], dtype).cpu().numpy()[0]
    tol = 1e-10 * max(1.0, np.sum(np.abs(w))) if dtype == "c128" else 1e-4 * np.maximum(1.0, np.abs(one))
    assert np.all(np.abs(row - one) <= tol), (row, one)
