"""complex128 and complex64 calls from |+> whose cost is symmetric (C(z) = C(~z)) sweep half the state; any
other cost sweeps all of it.  The choice is made on the device from C itself.

Tolerances: <C> and gradients within 1e-10 max(1, sum|w|) (complex128) or 1e-4 max(1, |value|)
(complex64), so two forms differ by at most twice that; states at n = 20 within 1e-11 or 1e-5 in
2-norm per pass.
"""
import numpy as np
import pytest

import synth
from oracle import qaoa

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


def problem(n, weights):
    e, w, integer = synth.graph("gnp", n, n, weights, prob=0.2)
    cv = q.cost_vector(q.Graph(n, e, w, integer), "i32" if integer else "f64")
    return cv, max(1.0, float(np.sum(np.abs(w))))


def tol(dtype, scale, ref):
    return 1e-10 * scale if dtype == "c128" else 1e-4 * np.maximum(1.0, np.abs(ref))


@pytest.mark.parametrize("n", [19, 20, 21, 22, 23, 24, 25, 26])
@pytest.mark.parametrize("weights", ["int", "u01"])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_half_against_whole(n, weights, dtype):
    cv, scale = problem(n, weights)
    gam, bet = synth.angles(3, n)
    psi, ref = q.new_state(n, dtype), q.new_state(n, dtype)
    out = q.apply_layers(psi, cv, gam, bet, expect=True).cpu().numpy()
    ref.fill_(2.0 ** (-0.5 * n))
    want = q.apply_layers(ref, cv, gam, bet, init=False, expect=True).cpu().numpy()  # a given state: all of it
    assert np.all(np.abs(out - want) <= 2 * tol(dtype, scale, want))
    # the adjoint pass's <C> is the forward pass's
    got = q.gradient(psi, ref, cv, gam, bet).cpu().numpy()
    assert np.all(np.abs(got[:2] - want) <= 2 * tol(dtype, scale, want))


@pytest.mark.parametrize("dtype,ts", [("c128", 1e-11), ("c64", 1e-5)])
@pytest.mark.parametrize("weights", ["int", "u01"])
@pytest.mark.parametrize("change", [None, 0, 5, (1 << 19) - 1, 1 << 19, (1 << 20) - 1])
def test_symmetry_is_read_from_the_cost(weights, change, dtype, ts):
    """One entry off anywhere: the whole call falls back; results are the oracle's either way."""
    n, p = 20, 2
    cv, scale = problem(n, weights)
    if change is not None:
        if weights == "int":  # within the descriptor's bounds
            cv.C[change] = cv.cmin + 1 if int(cv.C[change]) == cv.cmin else cv.cmin
        else:
            cv.C[change] += 1.0
    C = cv.C.cpu().numpy().astype(np.float64)
    gam, bet = synth.angles(p, 3)
    E, dg, db, _ = qaoa.adjoint_gradient(n, C, gam, bet)
    want = np.concatenate([[E, 1.0], dg, db])
    psi, lam = q.new_state(n, dtype), q.new_state(n, dtype)
    got = q.gradient(psi, lam, cv, gam, bet).cpu().numpy()
    assert np.all(np.abs(got - want) <= tol(dtype, scale, want))
    assert torch.linalg.vector_norm(psi - 2.0 ** (-0.5 * n)).item() <= 2 * ts  # the adjoint pass ends at |+>
    out = q.apply_layers(psi, cv, gam, bet, expect=True).cpu().numpy()
    assert np.all(np.abs(out - want[:2]) <= tol(dtype, scale, want[:2]))
    ref = qaoa.qaoa_state(n, C, gam, bet)
    assert np.linalg.norm(psi.cpu().numpy().astype(np.complex128) - ref) <= ts
