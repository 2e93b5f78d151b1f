"""Draws do not depend on the scale of the state: powers of two, from scales that the float32 search
of an eighth takes to those it leaves to float64 (masses outside 2^-60 .. 2^60, components outside
float32's range), give the same samples."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2407_13012_gb300 as q  # noqa: E402


@pytest.mark.parametrize("dtype,shifts", [("c128", (-200, -100, -45, -20, 20, 45, 100, 200)), ("c64", (-45, -20, 20, 45))])
def test_scales(dtype, shifts):
    n = 13
    rng = np.random.default_rng(1)
    cv = q.cost_vector(q.Graph(n, synth.gnp_edges(n, 0.4, 1), None, True), "i32")
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi *= np.exp2(rng.integers(-9, 1, 1 << n))
    state = torch.as_tensor(psi).to(torch.complex128 if dtype == "c128" else torch.complex64).cuda()
    z0 = q.sample(state, cv, 50000, 9)[0].cpu()
    for s in shifts:
        assert torch.equal(q.sample(state * 2.0 ** s, cv, 50000, 9)[0].cpu(), z0), s


@pytest.mark.parametrize("dtype,line", [("c64", 32), ("c128", 512)])
def test_few_shots_of_a_large_state(dtype, line):
    """Below one shot per 256 (complex128: 16) leaves the leaves keep no eighths; the draws are those of a
    larger call (the shots' uniforms are a counter stream)."""
    n = 23  # 8192 leaves
    rng = np.random.default_rng(2)
    cv = q.cost_vector(q.Graph(n, synth.gnp_edges(n, 0.2, 1), None, True), "i32")
    state = torch.as_tensor(rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n))
    state = state.to(torch.complex64 if dtype == "c64" else torch.complex128).cuda()
    z = q.sample(state, cv, 20000, 9)[0].cpu()
    for shots in (1, line - 1, line, line + 1):
        assert torch.equal(q.sample(state, cv, shots, 9)[0].cpu(), z[:shots]), shots
