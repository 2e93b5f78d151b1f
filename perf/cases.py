"""Performance cases: the work a user of this simulator has it do, through the Python binding.

Every case is one call (or one short run of calls) of the public entry points on one
problem instance:

  eval       cost vector, p layers with fused <C>, bitstring samples: one small circuit as a
             notebook or a test runs it, where launches and latency count
  layers     p layers from |+> with fused <C> on a resident state (energy scans, scale sweeps)
  gradient   the adjoint gradient of <C> in all 2p angles (one training evaluation)
  sample     bitstrings drawn from a resident state, with their costs
  adam       the on-device angle optimiser, a small training run from the linear ramp
  batch      adjoint gradients of many small graphs in one call (dataset generation)
  xy_layers, xy_gradient
             the same on the Hamming-weight subspace with the ring XY mixer (balanced cuts)

Graphs are random 3-regular or G(n, prob) with integer weights (int32 costs, phase tables) or
U(0, 1) weights (float64 costs, computed phases); angles are U(0, pi).  A program that
simulates in complex64 keeps scalars (<C>, norm, gradients) in float32, which holds all of the
digits such a run has.

exact() recomputes every float output in 64 bits with plain torch, one qubit or pair gate at a
time, without the package.
"""
import math

import numpy as np
import torch

import paper_2407_13012_gb300 as q

DEV = "cuda"


# ------------------------------------------------------------------------------- the cases


def listed():
    return [
        # a first small circuit: n = 10, G(10, 0.5), unit weights, p = 2, 4096 shots
        {"name": "eval_n10", "kind": "eval", "n": 10, "p": 2, "dtype": "c128", "weights": "unit", "prob": 0.5,
         "shots": 4096},
        # training a small instance on the device: 50 Adam steps at n = 14, p = 4
        {"name": "adam_n14", "kind": "adam", "n": 14, "p": 4, "dtype": "c128", "weights": "int", "prob": 0.3,
         "steps": 50},
        # an ordinary circuit: 3-regular, integer weights, n = 20, p = 8
        {"name": "layers_n20_c128", "kind": "layers", "n": 20, "p": 8, "dtype": "c128", "weights": "int", "prob": 0.0},
        # the large complex128 circuit: 16 GB of state, 3-regular, p = 6
        {"name": "layers_n30_c128", "kind": "layers", "n": 30, "p": 6, "dtype": "c128", "weights": "int", "prob": 0.0},
        # single precision, odd n, U(0, 1) weights (computed phases)
        {"name": "layers_n29_c64_u01", "kind": "layers", "n": 29, "p": 5, "dtype": "c64", "weights": "u01",
         "prob": 0.1},
        # deep training evaluation with U(0, 1) weights on a denser graph
        {"name": "grad_n24_c128_u01", "kind": "gradient", "n": 24, "p": 10, "dtype": "c128", "weights": "u01",
         "prob": 0.2},
        # large training evaluation, complex128
        {"name": "grad_n28_c128", "kind": "gradient", "n": 28, "p": 6, "dtype": "c128", "weights": "int", "prob": 0.0},
        # large training evaluation, complex64
        {"name": "grad_n30_c64", "kind": "gradient", "n": 30, "p": 3, "dtype": "c64", "weights": "int", "prob": 0.0},
        # a million shots from a large state
        {"name": "sample_n28_c128", "kind": "sample", "n": 28, "dtype": "c128", "shots": 1000000},
        # thousands of small graphs of uneven n, half 3-regular, half G(n, 0.3)
        {"name": "batch_4096_c128", "kind": "batch", "graphs": 4096, "n_lo": 8, "n_hi": 20, "p": 3, "dtype": "c128",
         "weights": "int", "prob": 0.3},
        # balanced cut on the feasible subspace: binom(30, 15) = 1.55e8 amplitudes
        {"name": "xy_layers_n30_c128", "kind": "xy_layers", "n": 30, "k": 15, "p": 3, "dtype": "c128",
         "weights": "int", "prob": 0.0},
        # a subspace training evaluation off the balanced point, odd n, single precision
        {"name": "xy_grad_n27_c64", "kind": "xy_gradient", "n": 27, "k": 12, "p": 2, "dtype": "c64",
         "weights": "int", "prob": 0.2},
    ]


def draw(rng):
    """One more case: the kinds in proportion to the listed ones, sizes over the same ranges, and
    no more work than the largest listed cases (a complex128 layer at n = 30 is 2^30 units; a
    gradient layer costs about four, a computed phase half as much again)."""
    kind = rng.choice(["eval", "adam", "layers", "layers", "layers", "gradient", "gradient", "gradient", "sample",
                       "batch", "xy_layers", "xy_gradient"])
    c = {"kind": kind, "dtype": rng.choice(["c128", "c128", "c64"]), "weights": rng.choice(["int", "int", "u01"])}
    if kind == "eval":  # shots depend on the last bits of the state: complex128 only
        c.update(n=rng.randint(4, 14), p=rng.randint(1, 5), dtype="c128", weights=rng.choice(["unit", "int", "u01"]),
                 prob=rng.choice([0.3, 0.5, 0.7]), shots=int(2 ** rng.uniform(6, 12.5)))
    elif kind == "adam":
        c.update(n=rng.randint(6, 18), p=rng.randint(1, 6), dtype="c128", prob=rng.choice([0.3, 0.5]),
                 steps=rng.randint(10, 60))
    elif kind in ("layers", "gradient"):
        c["n"] = rng.randint(16, 30 if kind == "layers" else 29)
        unit = (1.0 if kind == "layers" else 4.0) * (1.5 if c["weights"] == "u01" else 1.0) * (
            0.6 if c["dtype"] == "c64" else 1.0)
        most = int(5 * 2.0 ** 30 / (unit * 2.0 ** c["n"]))
        if most < 1:
            c["n"] -= 2
            most = int(5 * 2.0 ** 30 / (unit * 2.0 ** c["n"]))
        c["p"] = rng.randint(1, max(1, min(most, 10)))
        c["prob"] = _family(rng, c["n"])
    elif kind == "sample":
        c.pop("weights")
        c.update(n=rng.randint(12, 29), shots=int(10 ** rng.uniform(3, 6)))
    elif kind == "batch":
        lo = rng.randint(6, 12)
        c.update(graphs=int(2 ** rng.uniform(5, 11.5)), n_lo=lo, n_hi=rng.randint(lo + 1, 20), p=rng.randint(1, 4),
                 prob=rng.choice([0.3, 0.5]))
    else:
        n = rng.randint(12, 29 if kind == "xy_layers" else 27)
        c.update(n=n, k=max(1, n // 2 - rng.randint(0, 3)), p=rng.randint(1, 3), prob=_family(rng, n))
    return c


def _family(rng, n):
    """0.0 stands for random 3-regular (even n), else the edge probability of G(n, prob)."""
    return 0.0 if n % 2 == 0 and rng.random() < 0.5 else rng.choice([0.1, 0.2])


# ------------------------------------------------------------------------------ the inputs


def _edges(rng, n, prob):
    if prob:
        u, v = np.triu_indices(n, k=1)
        keep = rng.random(len(u)) < prob
        if not keep.any():
            keep[0] = True
        return np.stack([u[keep], v[keep]], axis=1).astype(np.int32)
    while True:  # random 3-regular: pair up three half-edges per vertex until the graph is simple
        e = np.sort(rng.permutation(np.repeat(np.arange(n), 3)).reshape(-1, 2), axis=1)
        if (e[:, 0] != e[:, 1]).all() and len(set(map(tuple, e.tolist()))) == len(e):
            return e.astype(np.int32)


def _weights(rng, m, kind, hi=10):
    if kind == "unit":
        return np.ones(m)
    return rng.random(m) if kind == "u01" else rng.integers(1, hi + 1, m).astype(np.float64)


def _instance(case, seed):
    """(edges, weights, gammas, betas) of a one-graph case."""
    rng = np.random.default_rng([2407, seed])
    e = _edges(rng, case["n"], case["prob"])
    w = _weights(rng, len(e), case["weights"])
    a = rng.random((2, case["p"])) * math.pi
    return e, w, a[0].copy(), a[1].copy()


def _batch_instances(case, seed):
    """Lists of n, edges, weights, and the (graphs, 2p) angles: a fair coin between 3-regular
    (even n) and G(n, prob), integer weights {1..5} or U(0, 1)."""
    rng = np.random.default_rng([13012, seed])
    lo, hi = case["n_lo"], case["n_hi"]
    evens = [n for n in range(lo, hi + 1) if n % 2 == 0]
    ns, es, ws = [], [], []
    for _ in range(case["graphs"]):
        reg3 = bool(evens) and rng.random() < 0.5
        n = int(rng.choice(evens)) if reg3 else int(rng.integers(lo, hi + 1))
        e = _edges(rng, n, 0.0 if reg3 else case["prob"])
        ns.append(n)
        es.append(e)
        ws.append(_weights(rng, len(e), case["weights"], 5))
    return ns, es, ws, rng.random((case["graphs"], 2 * case["p"])) * math.pi


def _sample_state(case, seed):
    """A normalised random complex state, as deep circuits make it, and the graph of its costs."""
    g = torch.Generator(DEV).manual_seed(seed)
    real = torch.float64 if case["dtype"] == "c128" else torch.float32
    psi = torch.view_as_complex(torch.randn(1 << case["n"], 2, device=DEV, dtype=real, generator=g))
    psi /= math.sqrt(2.0 * (1 << case["n"]))
    rng = np.random.default_rng([299, seed])
    e = _edges(rng, case["n"], 0.3)
    return psi, e, _weights(rng, len(e), "int")


def _graph(n, e, w, weights):
    return q.Graph(n, e, None if weights == "unit" else w, weights != "u01")


def _cost_kind(case):
    return "f64" if case.get("weights") == "u01" else "i32"


def prepare(case, seed):
    s = {"case": case, "seed": seed}
    kind = case["kind"]
    if kind == "batch":
        ns, es, ws, s["angles"] = _batch_instances(case, seed)
        s["graphs"] = [_graph(n, e, w, case["weights"]) for n, e, w in zip(ns, es, ws)]
        return s
    if kind == "sample":
        s["psi"], e, w = _sample_state(case, seed)
        s["cost"] = q.cost_vector(_graph(case["n"], e, w, "int"), "i32")
        return s
    n = case["n"]
    e, w, s["gam"], s["bet"] = _instance(case, seed)
    s["graph"] = _graph(n, e, w, case["weights"])
    if kind == "eval":
        s["psi"] = q.new_state(n, case["dtype"])
        return s
    if kind in ("xy_layers", "xy_gradient"):
        s["cost"] = q.xy_cost_vector(s["graph"], case["k"], _cost_kind(case))
        s["psi"] = q.xy_new_state(n, case["k"], case["dtype"])
        if kind == "xy_gradient":
            s["lam"] = q.xy_new_state(n, case["k"], case["dtype"])
        return s
    s["cost"] = q.cost_vector(s["graph"], _cost_kind(case))
    if kind == "adam":
        s["start"] = torch.tensor(_adam_start(case, seed), device=DEV)
        return s
    s["psi"] = q.new_state(n, case["dtype"])
    if kind == "gradient":
        s["lam"] = q.new_state(n, case["dtype"])
    return s


def _adam_start(case, seed):
    """Starting angles near the linear ramp."""
    p = case["p"]
    i = np.arange(1, p + 1) / p
    return np.concatenate([0.3 * i, 0.6 * (1.1 - i)]) + 0.05 * np.random.default_rng([7, seed]).random(2 * p)


def _scalars(out, case):
    return out.float() if case["dtype"] == "c64" else out


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "eval":
        cost = q.cost_vector(s["graph"], _cost_kind(case))
        out = q.apply_layers(s["psi"], cost, s["gam"], s["bet"], expect=True)
        z, cz = q.sample(s["psi"], cost, case["shots"], s["seed"])
        return {"C": cost.C, "psi": s["psi"], "expect": out, "z": z, "cz": cz}
    if kind == "layers":
        out = q.apply_layers(s["psi"], s["cost"], s["gam"], s["bet"], expect=True)
        return {"psi": s["psi"], "expect": _scalars(out, case)}
    if kind == "gradient":
        return {"grad": _scalars(q.gradient(s["psi"], s["lam"], s["cost"], s["gam"], s["bet"]), case)}
    if kind == "sample":
        z, cz = q.sample(s["psi"], s["cost"], case["shots"], s["seed"])
        return {"z": z, "cz": cz}
    if kind == "adam":
        angles = s["start"].clone()
        hist = q.optimize_adam(s["cost"], angles, case["steps"], lr=0.02, dtype=case["dtype"])
        return {"angles": angles, "history": hist}
    if kind == "batch":
        return {"grad": _scalars(q.batch_gradient(s["graphs"], s["angles"], case["dtype"]), case)}
    n, k = case["n"], case["k"]
    if kind == "xy_layers":
        out = q.xy_apply_layers(s["psi"], n, k, s["cost"], s["gam"], s["bet"], expect=True)
        return {"psi": s["psi"], "expect": _scalars(out, case)}
    return {"grad": _scalars(q.xy_gradient(s["psi"], s["lam"], n, k, s["cost"], s["gam"], s["bet"]), case)}


# ----------------------------------------------------------------------------- its least work


def work(case):
    """Inputs read once, outputs written once; operations of p layers with 6 per amplitude and
    RX gate (a complex combination of two amplitudes) and 6 per phase, three times that for a
    gradient (forward, and both states undone) plus the 4-operation terms of each gate."""
    kind = case["kind"]
    S = 16 if case["dtype"] == "c128" else 8
    cb = 8 if case.get("weights") == "u01" else 4
    if kind == "sample":
        return {"bytes": (1 << case["n"]) * S + case["shots"] * (16 + cb), "flops": 4.0 * (1 << case["n"])}
    p = case["p"]
    if kind == "batch":
        lo, hi = case["n_lo"], case["n_hi"]
        evens = [n for n in range(lo, hi + 1) if n % 2 == 0]
        share = 0.5 if evens else 0.0
        dist = [(n, (share / len(evens) if n in evens else 0.0) + (1 - share) / (hi - lo + 1))
                for n in range(lo, hi + 1)]
        f = case["graphs"] * sum(x * (1 << n) * p * (22 * n + 18) for n, x in dist)
        m = case["graphs"] * sum(x * 1.5 * n for n, x in dist)
        return {"bytes": 16 * m + case["graphs"] * 8 * (4 * p + 2), "flops": float(f)}
    n = case["n"]
    size = math.comb(n, case["k"]) if "k" in case else 1 << n
    # a ring pair gate moves the states whose two bits differ
    gate = n * (2.0 * math.comb(n - 2, case["k"] - 1) / size if "k" in case else 1.0)
    fwd, back = p * size * (6 * gate + 6), p * size * (16 * gate + 16)
    if kind == "eval":
        return {"bytes": size * (S + cb) + case["shots"] * 16, "flops": fwd}
    if kind in ("layers", "xy_layers"):
        return {"bytes": size * (S + cb), "flops": fwd}
    if kind == "adam":
        return {"bytes": size * cb + 8 * case["steps"] * (4 * p + 2), "flops": case["steps"] * (fwd + back)}
    return {"bytes": size * cb + 8 * (2 * p + 2), "flops": fwd + back}


# ------------------------------------------------------- the same in 64 bits, plainly in torch

CHUNK = 1 << 25


def _cuts(n, e, w, z=None):
    """C(z) in float64, of all 2^n z or of the given ones."""
    size = 1 << n if z is None else len(z)
    C = torch.zeros(size, dtype=torch.float64, device=DEV)
    for lo in range(0, size, CHUNK):
        hi = min(size, lo + CHUNK)
        x = torch.arange(lo, hi, dtype=torch.int64, device=DEV) if z is None else z[lo:hi].to(torch.int64)
        for (u, v), wt in zip(e.tolist(), w.tolist()):
            C[lo:hi] += wt * (((x >> u) ^ (x >> v)) & 1).to(torch.float64)
    return C


def _phase(psi, C, gamma):
    """psi (B, N) *= exp(-i gamma C), gamma (B,)."""
    for lo in range(0, psi.shape[1], max(1, CHUNK // psi.shape[0])):
        sl = slice(lo, lo + max(1, CHUNK // psi.shape[0]))
        a = C[:, sl] * -gamma[:, None]
        psi[:, sl] *= torch.complex(torch.cos(a), torch.sin(a))


def _rx_all(psi, n, beta):
    """RX(2 beta) on every qubit of each row."""
    B = psi.shape[0]
    c = torch.cos(beta).to(torch.complex128).view(B, 1, 1)
    ms = (-1j * torch.sin(beta)).view(B, 1, 1)
    for j in range(n):
        v = psi.view(B, -1, 2, 1 << j)
        a, b = v[:, :, 0], v[:, :, 1]
        t = a * c
        t.addcmul_(b, ms)
        b.mul_(c).addcmul_(a, ms)
        a.copy_(t)


def _sums(x):
    return x.reshape(x.shape[0], -1).sum(1)


def _dot(a, b):
    return _sums(a.conj() * b)


def _diag(psi, C, lam=None):
    """Per row, chunked: sum C |psi|^2 (real), or <lam|C|psi>."""
    total = 0
    step = max(1, CHUNK // psi.shape[0])
    for lo in range(0, psi.shape[1], step):
        sl = slice(lo, lo + step)
        x = psi[:, sl]
        total = total + (_sums(C[:, sl] * (x.real ** 2 + x.imag ** 2)) if lam is None
                         else _sums(C[:, sl] * (lam[:, sl].conj() * x)))
    return total


def _ones(psi):
    return torch.ones(1, 1, dtype=torch.float64, device=DEV).expand(psi.shape)


def _forward(n, C, gam, bet):
    psi = torch.full(C.shape, 2.0 ** (-n / 2), dtype=torch.complex128, device=DEV)
    for g, b in zip(gam.T, bet.T):
        _phase(psi, C, g)
        _rx_all(psi, n, b)
    return psi


def _expect(psi, C):
    return torch.stack([_diag(psi, C), _diag(psi, _ones(psi))], 1)


def _gradient(n, C, gam, bet):
    """Rows [E, norm, dE/dgamma, dE/dbeta] for C (B, 2^n), gam and bet (B, p)."""
    psi = _forward(n, C, gam, bet)
    out = _expect(psi, C)
    lam = psi * C
    dg, db = torch.zeros_like(gam), torch.zeros_like(bet)
    B = psi.shape[0]
    for l in reversed(range(gam.shape[1])):
        for j in range(n):
            x, y = psi.view(B, -1, 2, 1 << j), lam.view(B, -1, 2, 1 << j)
            db[:, l] += 2 * (_dot(y[:, :, 0], x[:, :, 1]) + _dot(y[:, :, 1], x[:, :, 0])).imag
        for s in (psi, lam):
            _rx_all(s, n, -bet[:, l])
        dg[:, l] = 2 * _diag(psi, C, lam).imag
        for s in (psi, lam):
            _phase(s, C, -gam[:, l])
    return torch.cat([out, dg, db], 1)


def _subspace(n, k):
    """Every z of popcount k, increasing."""
    parts = []
    for lo in range(0, 1 << n, CHUNK):
        z = torch.arange(lo, min(1 << n, lo + CHUNK), dtype=torch.int64, device=DEV)
        c = sum(((z >> i) & 1) for i in range(n))
        parts.append(z[c == k])
    return torch.cat(parts).to(torch.int32)


def _ring(n, z):
    """The ring's pairs in parity order, each as the two index lists that the gate mixes."""
    pairs = [(j, j + 1) for j in range(0, n - 1, 2)] + [(j, j + 1) for j in range(1, n - 1, 2)]
    gates = []
    for a, b in pairs + ([(0, n - 1)] if n > 2 else []):
        i = torch.nonzero(((z >> a) & 1 == 1) & ((z >> b) & 1 == 0)).view(-1)
        gates.append((i.to(torch.int32), torch.searchsorted(z, (z[i] - (1 << a) + (1 << b)), out_int32=True)))
    return gates


def _xy_gate(psi, i, j, beta):
    c, ms = math.cos(beta), -1j * math.sin(beta)
    a, b = psi[i], psi[j]
    psi[i] = c * a + ms * b
    psi[j] = c * b + ms * a


def _xy(case, seed):
    n, k = case["n"], case["k"]
    e, w, gam, bet = _instance(case, seed)
    z = _subspace(n, k)
    C = _cuts(n, e, w, z)[None]
    gates = _ring(n, z)
    psi = torch.full(C.shape, 1.0 / math.sqrt(C.shape[1]), dtype=torch.complex128, device=DEV)
    g = torch.tensor(gam, device=DEV)[:, None]
    for l in range(case["p"]):
        _phase(psi, C, g[l])
        for i, j in gates:
            _xy_gate(psi[0], i, j, bet[l])
    out = _expect(psi, C)
    if case["kind"] == "xy_layers":
        return {"psi": psi[0], "expect": out[0]}
    lam = psi * C
    dg, db = torch.zeros(2, case["p"], dtype=torch.float64, device=DEV)
    for l in reversed(range(case["p"])):
        for i, j in reversed(gates):
            db[l] += 2 * (torch.vdot(lam[0][i], psi[0][j]) + torch.vdot(lam[0][j], psi[0][i])).imag
            for s in (psi, lam):
                _xy_gate(s[0], i, j, -bet[l])
        dg[l] = 2 * _diag(psi, C, lam).imag[0]
        for s in (psi, lam):
            _phase(s, C, -g[l])
    return {"grad": torch.cat([out[0], dg, db])}


def _adam(case, seed):
    n, p, steps = case["n"], case["p"], case["steps"]
    e, w, _, _ = _instance(case, seed)
    C = _cuts(n, e, w)[None]
    x = torch.tensor(_adam_start(case, seed), device=DEV)
    m, v = torch.zeros_like(x), torch.zeros_like(x)
    rows = []
    for t in range(1, steps + 1):
        r = _gradient(n, C, x[None, :p], x[None, p:])[0]
        rows.append(torch.cat([r, x]))
        m = 0.9 * m + 0.1 * r[2:]
        v = 0.999 * v + 0.001 * r[2:] ** 2
        x = x + 0.02 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return {"angles": x, "history": torch.stack(rows)}


def _batch(case, seed):
    ns, es, ws, ang = _batch_instances(case, seed)
    p = case["p"]
    out = torch.zeros(len(ns), 2 * p + 2, dtype=torch.float64, device=DEV)
    a = torch.tensor(ang, device=DEV)
    for n in sorted(set(ns)):
        rows = [i for i, m in enumerate(ns) if m == n]
        at = max(1, (1 << 27) >> n)
        for lo in range(0, len(rows), at):
            part = rows[lo:lo + at]
            idx = torch.tensor(part, device=DEV)
            # all cuts of these graphs at once: a (graphs, pairs) weight matrix times the pair parities
            u, v = np.triu_indices(n, k=1)
            W = np.zeros((len(part), n, n))
            for r, i in enumerate(part):
                W[r, es[i][:, 0], es[i][:, 1]] = ws[i]
            W = torch.tensor(W[:, u, v], device=DEV)
            z = torch.arange(1 << n, device=DEV)
            C = torch.zeros(len(part), 1 << n, dtype=torch.float64, device=DEV)
            for c, (i, j) in enumerate(zip(u.tolist(), v.tolist())):
                C.addcmul_(W[:, c:c + 1], (((z >> i) ^ (z >> j)) & 1).to(torch.float64)[None])
            out[idx] = _gradient(n, C, a[idx, :p], a[idx, p:])
    return {"grad": out}


def exact(case, seed):
    """What run() returns, in 64 bits; None for drawn bitstrings, which have no such value."""
    kind = case["kind"]
    if kind == "sample":
        return None
    if kind == "batch":
        return _batch(case, seed)
    if kind == "adam":
        return _adam(case, seed)
    if kind in ("xy_layers", "xy_gradient"):
        return _xy(case, seed)
    n = case["n"]
    e, w, gam, bet = _instance(case, seed)
    C = _cuts(n, e, w)[None]
    g, b = torch.tensor(gam, device=DEV)[None], torch.tensor(bet, device=DEV)[None]
    if kind == "gradient":
        return {"grad": _gradient(n, C, g, b)[0]}
    psi = _forward(n, C, g, b)
    out = {"psi": psi[0], "expect": _expect(psi, C)[0]}
    if kind == "eval":
        out.update(C=C[0] if case["weights"] == "u01" else None, z=None, cz=None)
    return out
