"""complex64 computed phases keep float32's relative precision down to the smallest turns: one layer
without a mixer leaves -sin(gamma C) 2^(-n/2) in the imaginary parts.  Each is within 8 x 2^-24 relative
for small angles: the turn (1/2 ulp), sine (2), the amplitude and the product (1/2 each), with room.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


@pytest.mark.parametrize("n", [10, 16, 22])
@pytest.mark.parametrize("gamma", [1e-2, -1e-3, 1e-5, 1e-7, -1e-8, 1e-10, 1e-16, 1e-30])
def test_small_phases(n, gamma):
    e, w, integer = synth.graph("gnp", n, n, "u01", prob=0.3)
    cv = q.cost_vector(q.Graph(n, e, w, integer), "f64")
    psi = q.new_state(n, "c64")
    q.apply_layers(psi, cv, [gamma], [0.0])
    want = -torch.sin(gamma * cv.C) * 2.0 ** (-0.5 * n)
    got = psi.imag.double()
    assert torch.all((got - want).abs() <= 8 * 2.0 ** -24 * want.abs())
