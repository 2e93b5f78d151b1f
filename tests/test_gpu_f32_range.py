"""complex64 reductions beyond float32's range.  A state of huge norm has <C> and a norm^2 that float64 holds
and float32 does not: they are returned as float64 sums of the threads' float32 sums, within 1e-5 of the
sums over the state read back (32 float32 additions per thread), and infinite sums are infinite.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


def run(n, weights, amp):
    e, w, integer = synth.graph("gnp", n, n, weights, prob=0.3)
    w = np.asarray(w) * 1e5
    cv = q.cost_vector(q.Graph(n, e, w, integer), "i32" if integer else "f64")
    gam, bet = synth.angles(2, n)
    psi = q.new_state(n, "c64")
    psi.fill_(amp)
    out = q.apply_layers(psi, cv, np.asarray(gam) * 1e-5, bet, init=False, expect=True).cpu().numpy()
    return out, psi, cv


@pytest.mark.parametrize("n", [10, 13, 16, 21])
@pytest.mark.parametrize("weights", ["int", "u01"])
@pytest.mark.parametrize("amp", [1e10, 1e14])
def test_large_norms(n, weights, amp):
    out, psi, cv = run(n, weights, amp)
    p2 = torch.view_as_real(psi).double().square().sum(1)
    want = np.array([(cv.C.double() * p2).sum().item(), p2.sum().item()])
    assert np.all(np.abs(out - want) <= 1e-5 * want)


@pytest.mark.parametrize("n", [10, 13, 16, 21])
@pytest.mark.parametrize("weights", ["int", "u01"])
def test_infinite_sums(n, weights):
    out, _, _ = run(n, weights, 1e18)  # |psi|^2 C is above 1e41
    assert out[0] == np.inf


def test_gradient_of_large_costs():
    """dE/dbeta of costs near 1e37 passes float32 where its threads' sums do not: it scales with the costs."""
    n, f = 20, 1e36
    e, w, integer = synth.graph("gnp", n, n, "u01", prob=0.3)
    gam, bet = synth.angles(1, n)
    out = []
    for s in (1.0, f):
        cv = q.cost_vector(q.Graph(n, e, np.asarray(w) * s, False), "f64")
        psi, lam = q.new_state(n, "c64"), q.new_state(n, "c64")
        out.append(q.gradient(psi, lam, cv, np.asarray(gam) / s, bet).cpu().numpy())
    S = float(np.sum(w))
    assert abs(out[1][0] / f - out[0][0]) <= 1e-4 * S
    assert abs(out[1][3] / f - out[0][3]) <= 1e-4 * n * S
