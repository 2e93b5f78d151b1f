"""Sampling inside a leaf (GPU): the draw starts at the eighth of a 1024-entry leaf that its
running sums point to.  Mass next to eighth and leaf boundaries, empty eighths, a state the
16-byte loads cannot take, and a random state, each against the oracle on the same uniforms."""
import numpy as np
import pytest

import synth
from oracle import qaoa

pytestmark = pytest.mark.gpu


def _state(kind, n, rng):
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    if kind == "edges":  # only the entries on both sides of every eighth
        k = np.arange(1 << n) % 128
        psi[(k > 1) & (k < 126)] = 0
    elif kind == "gaps":  # whole eighths without mass, the last ones among them
        psi.reshape(-1, 128)[rng.random((1 << n) // 128) < 0.6] = 0
        psi[-256:] = 0
        psi[:2] = 1
    elif kind == "one":
        psi[:] = 0
        psi[(1 << n) - 129] = 1
    return psi / np.linalg.norm(psi)


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("kind", ["random", "edges", "gaps", "one", "unaligned"])
@pytest.mark.parametrize("n", [10, 13])
def test_eighths(dtype, kind, n):
    import torch
    import paper_2407_13012_gb300 as q
    if kind == "unaligned" and dtype == "c128":
        pytest.skip("complex128 entries are 16 bytes")
    rng = np.random.default_rng(n)
    edges = synth.gnp_edges(n, 0.4, 1)
    cv = q.cost_vector(q.Graph(n, edges, None, True), "i32")
    td = torch.complex128 if dtype == "c128" else torch.complex64
    host = torch.as_tensor(_state(kind, n, rng)).to(td)
    buf = torch.zeros((1 << n) + 1, dtype=td, device="cuda")
    psi = buf[1:] if kind == "unaligned" else buf[:-1]
    psi.copy_(host)
    z, cz = q.sample(psi, cv, 20000, 5)
    z = z.cpu().numpy()
    C = cv.C.cpu().numpy()
    ref, _ = qaoa.sample(host.numpy().astype(np.complex128), C, synth.sample_uniforms(5, 20000))
    # a target within rounding (~1e-13) of one of at most 2^13 steps: expected 2e-5 shots in all
    assert np.array_equal(z, ref.astype(np.int64))
    assert np.array_equal(cz.cpu().numpy(), C[z].astype(np.float64))
