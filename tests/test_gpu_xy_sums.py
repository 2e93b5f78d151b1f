"""complex64 subspace gradients: E, the norm and the gamma terms are sums over float32 states, formed
without rounding their terms to float32.  The state is read back and the same sums are taken in
float64, so only the summation differs: 1e-13 of sum|w| for E, 1e-14 for the norm (float64 sums of at
most 10^7 terms), and 1e-12 of sum|w|^2 for the gamma terms (double-float sums).
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


def problem(n, k, weights, scale):
    e, w, integer = synth.graph("gnp", n, n, weights, prob=0.3)
    w = np.asarray(w, dtype=np.float64) * scale
    return q.xy_cost_vector(q.Graph(n, e, w, integer), k, "i32" if integer else "f64"), float(np.sum(np.abs(w)))


SHAPES = [(12, 6), (15, 7), (22, 11), (26, 13)]
COSTS = [("int", 1.0), ("int", 1e6), ("u01", 1.0)]  # integer costs on both sides of 2^24, float64 costs


@pytest.mark.parametrize("n,k", SHAPES)
@pytest.mark.parametrize("weights,scale", COSTS)
def test_energy_and_norm(n, k, weights, scale):
    cv, S = problem(n, k, weights, scale)
    gam, bet = synth.angles(2, n)
    gam = np.asarray(gam) / scale
    psi, lam = q.xy_new_state(n, k, "c64"), q.xy_new_state(n, k, "c64")
    q.xy_apply_layers(psi, n, k, cv, gam, bet)
    p2 = torch.view_as_real(psi).double().square().sum(1)
    got = q.xy_gradient(psi, lam, n, k, cv, gam, bet).cpu().numpy()
    assert abs(got[0] - (cv.C.double() * p2).sum().item()) <= 1e-13 * S
    assert abs(got[1] - p2.sum().item()) <= 1e-14


@pytest.mark.parametrize("n,k", SHAPES)
@pytest.mark.parametrize("weights,scale", COSTS)
def test_gamma_term(n, k, weights, scale):
    """p = 1 without a mixer: lambda = C psi, rounded to float32 once, is known exactly."""
    cv, S = problem(n, k, weights, scale)
    gam = [0.7 / scale]
    psi, lam = q.xy_new_state(n, k, "c64"), q.xy_new_state(n, k, "c64")
    q.xy_apply_layers(psi, n, k, cv, gam, [0.0])
    C = cv.C.double()
    v = torch.view_as_real(psi).clone()
    l = (C.to(torch.float32)[:, None] * v).double()  # noqa: E741
    v = v.double()
    want = 2.0 * (C * (l[:, 0] * v[:, 1] - l[:, 1] * v[:, 0])).sum().item()
    got = q.xy_gradient(psi, lam, n, k, cv, gam, [0.0]).cpu().numpy()
    assert abs(got[2] - want) <= 1e-12 * S * S
