"""complex128 layers that continue a given state accept any norm: the state is scaled by a power of two
on loading and scaled back by the sweep that stores it, whichever kernels run in between.  Norms on
both sides of a power of two (their square's exponent decides the scale), at sizes whose plans mix
the sweep kernels: one and two groups, small tiles, groups below three qubits, odd and even p.

Tolerances: the state is linear in its input, so 1e-11 per pass in 2-norm, <C> to 1e-10 max(1, sum|w|)
and the norm to 1e-10, each times the input's scale (its square for <C> and the norm).
"""
import numpy as np
import pytest

import synth
from oracle import qaoa

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


@pytest.mark.parametrize("norm", [0.3, 1.0 - 1e-12, 1.0, 5.0, 2.0 ** -40, 2.0 ** 31])
@pytest.mark.parametrize("p", [1, 2])
@pytest.mark.parametrize("n", [3, 9, 10, 11, 12, 13, 15, 19, 20])
def test_continue_from_any_norm(n, p, norm):
    e, w, integer = synth.graph("gnp", n, n, "int", prob=0.5 if n < 10 else 0.2)
    cv = q.cost_vector(q.Graph(n, e, w, integer), "i32")
    C = qaoa.cut_values(n, e, w)
    scale = max(1.0, float(np.sum(np.abs(w))))
    psi0 = synth.random_state(n, 7)
    psi0 = psi0 / np.linalg.norm(psi0) * norm
    gam, bet = synth.angles(p, n)
    psi = torch.as_tensor(psi0, dtype=torch.complex128).cuda()
    out = q.apply_layers(psi, cv, gam, bet, init=False, expect=True).cpu().numpy()
    ref = qaoa.qaoa_state(n, C, gam, bet, psi0=psi0)
    assert np.linalg.norm(psi.cpu().numpy() - ref) <= 1e-11 * norm * p
    assert abs(out[0] - qaoa.expectation(ref, C)) <= 1e-10 * scale * norm * norm
    assert abs(out[1] - qaoa.norm2(ref)) <= 1e-10 * norm * norm


@pytest.mark.parametrize("factor", [0.75, 3.0])
@pytest.mark.parametrize("dtype,n", [("c128", 21), ("c128", 22), ("c128", 23), ("c128", 25), ("c64", 27), ("c64", 28)])
def test_scaled_state_against_plus(dtype, n, factor):
    """|+> times a factor, continued, is the call from |+> times the factor: all of a given state against a
    half state.  complex128: per path 2e-11 in 2-norm at n = 24, growing by 2^(1/2) per qubit; complex64:
    1e-5 per pass, <C> to 1e-4 max(1, |<C>|)."""
    e, w, integer = synth.graph("gnp", n, n, "u01", prob=0.2)
    cv = q.cost_vector(q.Graph(n, e, w, integer), "f64")
    scale = max(1.0, float(np.sum(np.abs(w))))
    gam, bet = synth.angles(2, n)
    psi, ref = q.new_state(n, dtype), q.new_state(n, dtype)
    want = q.apply_layers(ref, cv, gam, bet, expect=True).cpu().numpy()
    psi.fill_(factor * 2.0 ** (-0.5 * n))
    out = q.apply_layers(psi, cv, gam, bet, init=False, expect=True).cpu().numpy() / factor ** 2
    to = 1e-10 * scale if dtype == "c128" else 1e-4 * np.maximum(1.0, np.abs(want))
    ts = 7.6e-11 * 2 ** (0.5 * max(0, n - 24)) if dtype == "c128" else 2e-5
    assert np.all(np.abs(out - want) <= 2 * to)
    assert torch.linalg.vector_norm(psi / factor - ref).item() <= 2 * ts
