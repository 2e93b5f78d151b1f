"""Launch timing reports the bytes of the form that ran: half of the state for a symmetric cost (and the
stores of the other half), all of it for any other cost, which only the device tells apart."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


def timed(call):
    q.timing_enable(True)
    try:
        q.timing_read()
        call()
        torch.cuda.synchronize()
        ms, launches, nbytes, dropped = q.timing_read()
    finally:
        q.timing_enable(False)
    assert dropped == 0 and launches[0] > 0
    return nbytes


@pytest.mark.parametrize("dtype,n,S", [("c128", 20, 16), ("c64", 21, 8)])
def test_layers(dtype, n, S):
    e, w, integer = synth.graph("gnp", n, n, "int", prob=0.3)
    cv = q.cost_vector(q.Graph(n, e, w, integer), "i32")
    gam, bet = synth.angles(2, n)
    psi = q.new_state(n, dtype)
    # two groups: |+> stored; the second group loaded and stored; the first again; two of them read C
    per = (S + 4) + (2 * S + 4) + 2 * S
    assert timed(lambda: q.apply_layers(psi, cv, gam, bet))[0] == (per + S) * 2 ** (n - 1)
    cv.C[3] += 1
    assert timed(lambda: q.apply_layers(psi, cv, gam, bet))[0] == per * 2 ** n


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_subspace(dtype):
    n, k = 26, 13
    e, w, integer = synth.graph("gnp", n, n, "u01", prob=0.3)
    cv = q.xy_cost_vector(q.Graph(n, e, w, integer), k, "f64")
    gam, bet = synth.angles(1, n)
    psi, lam = q.xy_new_state(n, k, dtype), q.xy_new_state(n, k, dtype)
    calls = (lambda: q.xy_apply_layers(psi, n, k, cv, gam, bet), lambda: q.xy_gradient(psi, lam, n, k, cv, gam, bet))
    half = [timed(c)[0] for c in calls]
    cv.C[5] = torch.nextafter(cv.C[5], torch.full_like(cv.C[5], 1e300))
    whole = [timed(c)[0] for c in calls]
    assert np.array_equal(whole, 2 * np.array(half))
