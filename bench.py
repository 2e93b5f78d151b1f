"""Benchmark: MaxCut QAOA on one GB300 (replicas on N GPUs).

One step is one pass of the whole hot path on a seeded synthetic instance:
cost vector C(z), p layers with fused <C>, sampling, and the adjoint gradient
(p forward layers + p uncompute layers).  value = QAOA layers applied per second
(3p per step), whole job over all ranks.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
                  [--n 30] [--dtype c128] [--p 6] [--shots 1000000] [--family reg3]

Under torchrun every rank runs an independent replica (the simulation does not
shard); timing is the max over ranks.  ``--impl reference`` times the FP64 CPU
oracle on a bounded sample of the same workload on the host cores.

Outside the timed step the line also carries: ``gradient`` (gradient evaluations per
second), ``batched`` (4096 small graphs in one batched call against one at a time),
``time_to_ratio`` (time for 256 graphs to reach an approximation ratio: batched or plain
optimiser, from the linear ramp or the learned proposer) and ``cpu_baseline`` (the oracle
on one core and on all host cores).  ``--workload batched|xy|ttr`` prints one of those
measurements, or the Hamming-weight-subspace workload, as a line of its own.
"""
from __future__ import annotations

import argparse
import ctypes as ct
import json
import os
import statistics
import subprocess
import sys
import time
from pathlib import Path

import numpy as np

ROOT = Path(__file__).resolve().parent
sys.path.insert(0, str(ROOT))

METRIC = "QAOA layer sweeps/s & HBM GB/s at n=28-32; grad evals/s; batched vs plain"


def emit(line: dict, a) -> None:
    """Print the result line; with --jsonl also append it, with host and time, to a log."""
    text = json.dumps(line)
    print(text, flush=True)
    if getattr(a, "jsonl", None):
        rec = dict(line)
        rec["host"] = {"cores": os.cpu_count(), "time": time.strftime("%Y-%m-%dT%H:%M:%S")}
        with open(a.jsonl, "a") as f:
            f.write(json.dumps(rec) + "\n")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=None, help="qubits (default 30; 32 for --workload xy)")
    ap.add_argument("--dtype", default="c128", choices=["c128", "c64"])
    ap.add_argument("--p", type=int, default=6)
    ap.add_argument("--shots", type=int, default=1_000_000)
    ap.add_argument("--family", default="reg3", choices=["reg3", "gnp"])
    ap.add_argument("--prob", type=float, default=0.1, help="edge probability of G(n, p) (--family gnp)")
    ap.add_argument("--weights", default="int", choices=["int", "u01"],
                    help="integer weights {1..10} (int32 costs) or U(0,1) float64 weights")
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-batched", action="store_true", help="skip the batched-vs-plain measurement")
    ap.add_argument("--batch-graphs", type=int, default=4096)
    ap.add_argument("--no-ttr", action="store_true", help="skip the time-to-ratio measurement")
    ap.add_argument("--no-autotune", action="store_true",
                    help="batched workload: the library's default tile per qubit count instead of the autotuner's")
    ap.add_argument("--ttr-graphs", type=int, default=256)
    ap.add_argument("--ttr-target", type=float, default=0.88)
    ap.add_argument("--jsonl", default=None, help="also append the JSON line to this file (a run log)")
    ap.add_argument("--workload", default="layers", choices=["layers", "batched", "xy", "ttr"],
                    help="layers: the n-qubit step (default); batched: only the batched-gradient workload; "
                         "xy: QAOA on the Hamming-weight-k subspace with the ring XY mixer (balanced cut); "
                         "ttr: only the time-to-ratio comparison of the optimisers")
    ap.add_argument("--k", type=int, default=None, help="Hamming weight of the xy workload (default n/2)")
    a = ap.parse_args()
    if a.n is None:
        a.n = 32 if a.workload == "xy" else 30
    if a.warmup < 3:
        a.warmup = 3
    return a


def workload_name(a):
    fam = "random 3-regular" if a.family == "reg3" else f"G(n,{a.prob:g})"
    w = "U(0,1) fp64 weights" if a.weights == "u01" else "integer weights {1..10}"
    return (f"MaxCut QAOA n={a.n} {fam}, {w}, p={a.p}, {a.dtype} statevector: cost vector + "
            f"{a.p} layers with <C> + {a.shots} samples + adjoint gradient (2p layers)")


# What the kernels compute in.  complex128 states are stored as float64 pairs but, inside a
# call, held and transformed as int64 fixed point with a fixed resolution of 2^-54 (Q54):
# an amplitude of magnitude 2^-15 (n = 30) carries ~39 significant bits, not float64's 53.
ARITHMETIC = {
    "c128": "int64 fixed point, value = integer x 2^-54 (Q54), inside each call; float64 pairs (complex128) "
            "in memory between calls; reductions as integer sums of up to 128 bits, converted to float64",
    "c64": "float32 (complex64 state), threads' float32 sums added up in double-float and float64",
}


def arith_dtype(state_dtype: str) -> str:
    return "int64" if state_dtype == "c128" else "f32"


def make_instance(a):
    import synth
    fam = "gnp" if (a.family == "reg3" and a.n % 2) else a.family  # 3-regular needs even n
    e, w, integer = synth.graph(fam, a.n, a.seed, weights=a.weights, prob=a.prob)
    gam, bet = synth.angles(a.p, a.seed)
    return e, w, integer, gam, bet


def reduce_max(x: float, device=None) -> float:
    """Max of a per-rank scalar over all ranks (identity without a process group)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(units_per_rank: float, world: int, seconds_max: float) -> float:
    """Whole-job throughput: every rank's units over the slowest rank's time (weak scaling)."""
    return world * units_per_rank / seconds_max


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


def measured_peak_hbm():
    p = ROOT / "MEASURED_PEAKS.json"
    try:
        d = json.loads(p.read_text())
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


SWEEP_SOURCES = ("sweep.cu", "sweeper.cuh", "lean_kernel.cuh", "lean_f1.cu", "lean_f1d.cu", "lean_f2.cu", "lean_x1.cu",
                 "lean_x2_mix.cu", "lean_x2_ops.cu", "lean_xm.cu", "lean_xt.cu", "tile_layout.cuh", "fixedpoint.cuh",
                 "internal.h", "capi.cu")


def sweep_source_hash() -> str:
    """Hash of the sources that define and plan the layer-sweep kernels (the traffic record
    is valid while they are unchanged)."""
    import hashlib
    h = hashlib.sha256()
    for name in SWEEP_SOURCES:
        f = ROOT / "paper_2407_13012_gb300" / "csrc" / name
        h.update(name.encode())
        h.update(f.read_bytes())
    return h.hexdigest()[:16]


def traffic_record(kernel_hash: str, key: str):
    """Per-launch DRAM bytes of the sweep kernels for workload `key` from the committed ncu
    summary, if it was taken on the current sweep sources."""
    p = ROOT / "profiles" / "sweep_traffic.json"
    try:
        d = json.loads(p.read_text())
    except Exception:
        return None
    if d.get("source_hash") != kernel_hash:
        return None
    return d.get("workloads", {}).get(key)


# ------------------------------------------------------------------ CPU oracle baseline
#
# The oracle (numpy, as it stands) applies one full QAOA layer -- the phase on all 2^m
# amplitudes, then RX on each of the m qubits -- to the |+> state of the workload's graph
# family at a size m the host finishes in seconds.  It runs once on one core, then as
# independent copies on all cores at the same time (one process each, started with
# `spawn`, released together by a barrier): layers/s on the host = copies / wall time.
# Both rates are measured; the workload's n-qubit rate is their extrapolation by the
# layer's work, 2^(n - m) n / m (amplitudes x qubit passes), and the line says so.

def cpu_model() -> str:
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.split(":")[0].strip() == "Model name":
                return line.split(":", 1)[1].strip()
    except Exception:
        pass
    import platform
    return platform.processor() or platform.machine()


def _oracle_layer_child(m, family, weights, prob, seed, p, barrier, results):
    """One full oracle layer at m qubits; puts (start, end) wall-clock times on `results`."""
    import synth
    from oracle import qaoa
    fam = "gnp" if (family == "reg3" and m % 2) else family
    e, w, integer = synth.graph(fam, m, seed, weights=weights, prob=prob)
    gam, bet = synth.angles(p, seed)
    C = qaoa.cut_values(m, e, w, integer=integer)
    psi = qaoa.plus_state(m)
    barrier.wait()
    t0 = time.time()
    psi = qaoa.apply_cost_unitary(psi, C, gam[0])
    psi = qaoa.apply_rx_all(psi, m, bet[0])
    results.put((t0, time.time()))


def oracle_layers(a, m: int, copies: int):
    """Wall time of `copies` concurrent full oracle layers at m qubits (one process each)."""
    import multiprocessing as mp
    ctx = mp.get_context("spawn")
    barrier = ctx.Barrier(copies)
    results = ctx.Queue()
    procs = [ctx.Process(target=_oracle_layer_child, args=(m, a.family, a.weights, a.prob, a.seed, a.p, barrier,
                                                          results)) for _ in range(copies)]
    for pr in procs:
        pr.start()
    spans = [results.get() for _ in procs]
    for pr in procs:
        pr.join()
    return max(t1 for _, t1 in spans) - min(t0 for t0, _ in spans)


def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count() or 1


def cpu_baseline(a, m: int = 24):
    """The oracle's layer rate on the host: measured at m qubits on one core and on all
    cores, extrapolated to the workload's n qubits."""
    cores = min(host_cores(), 16)  # each copy holds ~1 GB at m = 24
    t1 = oracle_layers(a, m, 1)
    tall = oracle_layers(a, m, cores)
    scale = 2.0 ** (a.n - m) * a.n / m
    rate_all = cores / tall
    return {"value": rate_all / scale, "unit": "layers/s", "cores": cores, "kind": "oracle",
            "extrapolated": True, "scale": scale,
            "measured": {"m": m, "layer_s_one_core": t1, "layers_per_s_one_core": 1.0 / t1,
                         "layers_per_s_all_cores": rate_all, "copies": cores},
            "cpu_model": cpu_model(), "nproc": os.cpu_count(),
            "sample": (f"numpy oracle: one full layer (phase + RX on all {m} qubits) of the workload's graph family "
                       f"at m={m}, timed on 1 core ({t1:.2f} s) and as {cores} concurrent copies on {cores} cores "
                       f"({tall:.2f} s wall); layers/s extrapolated to n={a.n} by 2^(n-m) n/m = x{scale:.1f}")}


def run_reference(a, m: int = 22):
    """The oracle as the reference arm: each step is one round of concurrent full layers at
    m qubits on all host cores; layers/s extrapolated to the workload by 2^(n-m) n/m."""
    world, rank, local = dist_env()
    if rank != 0:
        return 0
    cores = min(host_cores(), 16)
    scale = 2.0 ** (a.n - m) * a.n / m
    walls = []
    for i in range(a.warmup + a.steps):
        wall = oracle_layers(a, m, cores)
        if i >= a.warmup:
            walls.append(wall)
    wall = statistics.mean(walls)
    value = cores / wall / scale            # workload layers per second on the host
    step = 3 * a.p / value                  # one step = 3p layer applications
    line = {"metric": METRIC, "impl": "reference", "value": value, "unit": "layers/s", "n_gpus": a.gpus,
            "steps": a.steps, "warmup": a.warmup, "ms_per_step": step * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": workload_name(a), "n": a.n, "p": a.p, "state_dtype": a.dtype},
            "cpu_baseline": {"value": value, "unit": "layers/s", "cores": cores, "kind": "oracle",
                             "extrapolated": True, "scale": scale, "cpu_model": cpu_model(),
                             "nproc": os.cpu_count(),
                             "sample": f"each step: {cores} concurrent full numpy-oracle layers at m={m} qubits "
                                       f"({wall:.2f} s wall), extrapolated to n={a.n} by 2^(n-m) n/m = x{scale:.1f}; "
                                       f"3p layers per step"},
            "e2e": {"value": value, "unit": "layers/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    emit(line, a)
    return 0


# ------------------------------------------------------------------ batched vs plain

BATCH_WORKLOAD = ("{g} graphs, n ~ U{{8..20}}, half random 3-regular / half G(n,0.3), integer weights {{1..5}}, "
                  "p=3, own angles per graph: <C> + adjoint gradient of every graph")


def measure_batched(q, dev, dtype: str, count: int, reps: int = 3, autotune: bool = True):
    """The batched workload: one batched call over all graphs against the plain path
    (cost vector + gradient per graph, one graph at a time), both timed with CUDA events."""
    import torch
    import synth
    p = 3
    insts = synth.batch_instances(count, 1, p=p)
    graphs = [q.Graph(n, e, w, True) for (n, f, e, w, g, b) in insts]
    ang = np.stack([np.concatenate([g, b]) for (*_, g, b) in insts])
    # tile size per qubit count from the autotuner, or the library's default choice
    tiles = q.batch_autotune(dtype, p, 8, 20, graphs_per_n=152, device=dev)[0] if autotune else None
    q.batch_gradient(graphs, ang, dtype, tiles=tiles, device=dev)
    torch.cuda.synchronize()
    ts = []
    for _ in range(reps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        out = q.batch_gradient(graphs, ang, dtype, tiles=tiles, device=dev)
        e1.record()
        torch.cuda.synchronize()
        ts.append(e0.elapsed_time(e1))
    batched_ms = statistics.median(ts)

    def plain(sub):
        res = []
        for gph, (n, f, e, w, g, b) in sub:
            cv = q.cost_vector(gph, "i32", device=dev)
            psi, lam = q.new_state(n, dtype, dev), q.new_state(n, dtype, dev)
            res.append(q.gradient(psi, lam, cv, g, b))
        return res

    pairs = list(zip(graphs, insts))
    plain(pairs[:64])
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    res = plain(pairs)
    e1.record()
    torch.cuda.synchronize()
    plain_ms = e0.elapsed_time(e1)
    agree = float(np.max(np.abs(out.cpu().numpy() - torch.stack(res).cpu().numpy())))
    return {"workload": BATCH_WORKLOAD.format(g=count), "state_dtype": dtype,
            "graph_grads_per_s": count / (batched_ms / 1e3), "batched_ms": batched_ms, "plain_ms": plain_ms,
            "speedup": plain_ms / batched_ms, "max_abs_diff_vs_plain": agree,
            "tiles": {int(n): int(tiles[n]) for n in range(8, 21)} if tiles is not None else "library default",
            "launches": "1 prep + grouped sweeps per size (n >= 16 c128, n >= 18 c64) + 1 persistent per tile size",
            "timing": "CUDA events, median of %d batched runs; plain: one run over all graphs" % reps}


TTR_WORKLOAD = ("{g} held-out graphs of the proposer family (G(n,0.3), n ~ U{{12..18}}, U(0,1) weights, seed 1002), "
                "p={p}; approximation ratio = <C> / max_z C(z); target ratio {r}")


def measure_time_to_ratio(q, dev, dtype: str = "c128", count: int = 256, target: float = 0.88,
                          max_steps: int = 300, lr: float = 0.03, max_evals: int = 60):
    """Time for every graph of a set to reach a fixed approximation ratio, four ways:
    plain (one graph at a time: cost vector + on-device L-BFGS, the paper's optimiser) or
    batched (all graphs per step in one persistent launch, Adam on the host between steps,
    graphs leave the batch once they reach the target), each from the linear ramp or from the
    learned proposer's angles (its inference inside the timed region).

    Host wall clock with the device synchronised.  plain: graphs run in order, so the time
    is that of every run before the last graph that reaches the target plus the share of that
    graph's run up to its first evaluation at the target (evaluations are equally long).
    batched: the step at which the last graph reaching the target reached it."""
    import torch
    import synth
    from paper_2407_13012_gb300 import proposer
    params, p, _ = proposer.load_weights()
    insts = synth.proposer_instances(count, 1002)
    graphs = [q.Graph(n, e, w, False) for n, e, w in insts]
    maxcut = np.array([float(q.cost_vector(g, "f64", device=dev).C.max().item()) for g in graphs])
    pt = torch.as_tensor(params, device=dev)
    q.propose_angles(graphs, pt, p, device=dev)  # warm-up of the inference kernel
    q.batch_gradient(graphs[:8], proposer.ramp_init(8, p), dtype, device=dev)
    torch.cuda.synchronize()

    def start_angles(kind):
        if kind == "ramp":
            return proposer.ramp_init(count, p)
        return q.propose_angles(graphs, pt, p, device=dev).cpu().numpy()

    def batched(kind):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ang = start_angles(kind)
        m, v = np.zeros_like(ang), np.zeros_like(ang)
        reached = np.full(count, np.nan)
        active = np.arange(count)
        steps = 0
        for t in range(1, max_steps + 1):
            out = q.batch_gradient([graphs[i] for i in active], ang[active], dtype, device=dev).cpu().numpy()
            steps = t
            hit = out[:, 0] / maxcut[active] >= target
            reached[active[hit]] = time.perf_counter() - t0
            keep = ~hit
            idx, g = active[keep], out[keep, 2:]
            m[idx] = 0.9 * m[idx] + 0.1 * g
            v[idx] = 0.999 * v[idx] + 0.001 * g * g
            ang[idx] += lr * (m[idx] / (1 - 0.9 ** t)) / (np.sqrt(v[idx] / (1 - 0.999 ** t)) + 1e-8)
            active = idx
            if len(active) == 0:
                break
        ok = ~np.isnan(reached)
        return {"reached": float(ok.mean()), "ms_to_ratio": float(np.max(reached[ok]) * 1e3) if ok.any() else None,
                "steps": steps}

    def plain(kind):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ang0 = start_angles(kind)
        elapsed = time.perf_counter() - t0
        at_last, evals, nreached = None, [], 0
        for i, g in enumerate(graphs):
            torch.cuda.synchronize()
            t1 = time.perf_counter()
            cv = q.cost_vector(g, "f64", device=dev)
            a = torch.as_tensor(ang0[i], device=dev)
            hist, info = q.optimize_lbfgs(cv, a, max_evals=max_evals, m=10, gtol=1e-6, dtype=dtype)
            best = np.maximum.accumulate(hist[:, 0].cpu().numpy()) / maxcut[i]
            wall = time.perf_counter() - t1
            hit = np.nonzero(best >= target)[0]
            if len(hit):
                k = int(hit[0]) + 1
                at_last = elapsed + wall * k / len(best)
                evals.append(k)
                nreached += 1
            elapsed += wall
        return {"reached": nreached / count, "ms_to_ratio": at_last * 1e3 if at_last is not None else None,
                "mean_evals_to_ratio": float(np.mean(evals)) if evals else None}

    res = {"workload": TTR_WORKLOAD.format(g=count, p=p, r=target), "state_dtype": dtype,
           "timing": "host wall clock, device synchronised; proposer inference inside the proposer arms",
           "batched": {"optimiser": f"Adam lr {lr}, at most {max_steps} steps, graphs leave once at the target"},
           "plain": {"optimiser": f"on-device L-BFGS (m = 10), at most {max_evals} evaluations per graph"}}
    for kind in ("ramp", "proposer"):
        res["plain"][kind] = plain(kind)
        res["batched"][kind] = batched(kind)
    base = res["plain"]["ramp"]["ms_to_ratio"]
    for arm in ("plain", "batched"):
        for kind in ("ramp", "proposer"):
            r = res[arm][kind]
            r["speedup_vs_plain_ramp"] = (base / r["ms_to_ratio"]) if (base and r["ms_to_ratio"]) else None
    return res


def measure_gradient(q, gradient_once, steps: int):
    """Gradient evaluations per second at the main configuration (CUDA events)."""
    import torch
    gradient_once()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(steps):
        gradient_once()
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / steps
    return {"evals_per_s": 1e3 / ms, "ms": ms}


# ------------------------------------------------------------------ GPU arm

def run_ours(a):
    import torch
    import torch.distributed as dist

    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    import paper_2407_13012_gb300 as q

    e, w, integer, gam, bet = make_instance(a)
    graph = q.Graph(a.n, e, w, integer)
    cdt = "i32" if integer else "f64"
    dev = torch.device("cuda", local)
    C = torch.empty(1 << a.n, dtype=torch.int32 if integer else torch.float64, device=dev)
    psi = q.new_state(a.n, a.dtype, dev)
    lam = q.new_state(a.n, a.dtype, dev)
    shots = a.shots
    z = torch.empty(shots, dtype=torch.int64, device=dev)
    cz = torch.empty(shots, dtype=torch.float64, device=dev)
    stream = torch.cuda.current_stream(dev)
    dt_code = q.C128 if a.dtype == "c128" else q.C64
    lo, hi = graph.check()
    span = hi - lo + 1 if integer else 0
    ws_bytes = max(q.workspace_size(a.n, dt_code, q.OP_LAYERS, a.p, 0, span),
                   q.workspace_size(a.n, dt_code, q.OP_SAMPLE, 0, shots),
                   q.workspace_size(a.n, dt_code, q.OP_GRADIENT, a.p, 0, span),
                   q.workspace_size(a.n, dt_code, q.OP_EXPECTATION))
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=dev)
    eout = torch.empty(2, dtype=torch.float64, device=dev)
    gout = torch.empty(2 * a.p + 2, dtype=torch.float64, device=dev)
    gp = gam.ctypes.data_as(ct.POINTER(ct.c_double))
    bp = bet.ctypes.data_as(ct.POINTER(ct.c_double))
    sp = ct.c_void_p(stream.cuda_stream)
    L = q.lib

    def chk(rc, what):
        if rc != 0:
            raise q.QaoaError(rc, what)

    def gradient_once():
        desc = q.CostT()
        gs = graph.as_struct()
        chk(L.qaoa_cost_vector(ct.byref(gs), ct.c_void_p(C.data_ptr()), q.COST_I32 if integer else q.COST_F64,
                               ct.byref(desc), sp), "cost")
        chk(L.qaoa_gradient(a.n, dt_code, ct.c_void_p(psi.data_ptr()), ct.c_void_p(lam.data_ptr()), ct.byref(desc),
                            gp, bp, a.p, ct.c_void_p(gout.data_ptr()), ct.c_void_p(ws.data_ptr()), ws_bytes, sp),
            "gradient")

    def step_device():
        desc = q.CostT()
        gs = graph.as_struct()
        chk(L.qaoa_cost_vector(ct.byref(gs), ct.c_void_p(C.data_ptr()), q.COST_I32 if integer else q.COST_F64,
                               ct.byref(desc), sp), "cost")
        chk(L.qaoa_apply_layers(a.n, dt_code, ct.c_void_p(psi.data_ptr()), ct.byref(desc), gp, bp, a.p, 1,
                                ct.c_void_p(eout.data_ptr()), ct.c_void_p(ws.data_ptr()), ws_bytes, sp), "layers")
        chk(L.qaoa_sample(a.n, dt_code, ct.c_void_p(psi.data_ptr()), ct.byref(desc), shots, 7,
                          ct.c_void_p(z.data_ptr()), ct.c_void_p(cz.data_ptr()), ct.c_void_p(ws.data_ptr()),
                          ws_bytes, sp), "sample")
        chk(L.qaoa_gradient(a.n, dt_code, ct.c_void_p(psi.data_ptr()), ct.c_void_p(lam.data_ptr()), ct.byref(desc),
                            gp, bp, a.p, ct.c_void_p(gout.data_ptr()), ct.c_void_p(ws.data_ptr()), ws_bytes, sp),
            "gradient")

    # host buffers for the end-to-end variant (pinned)
    z_host = torch.empty(shots, dtype=torch.int64, pin_memory=True)
    c_host = torch.empty(shots, dtype=torch.float64, pin_memory=True)
    g_host = np.zeros(2 * a.p + 2)
    e_host = np.zeros(2)

    def step_e2e():
        desc = q.CostT()
        gs = graph.as_struct()
        chk(L.qaoa_cost_vector(ct.byref(gs), ct.c_void_p(C.data_ptr()), q.COST_I32 if integer else q.COST_F64,
                               ct.byref(desc), sp), "cost")
        chk(L.qaoa_apply_layers(a.n, dt_code, ct.c_void_p(psi.data_ptr()), ct.byref(desc), gp, bp, a.p, 1, None,
                                ct.c_void_p(ws.data_ptr()), ws_bytes, sp), "layers")
        chk(L.qaoa_expectation_host(a.n, dt_code, ct.c_void_p(psi.data_ptr()), ct.byref(desc),
                                    e_host.ctypes.data_as(ct.POINTER(ct.c_double)), ct.c_void_p(ws.data_ptr()),
                                    ws_bytes, sp), "expectation_host")
        chk(L.qaoa_sample_host(a.n, dt_code, ct.c_void_p(psi.data_ptr()), ct.byref(desc), shots, 7,
                               ct.c_void_p(z.data_ptr()), ct.c_void_p(cz.data_ptr()), ct.c_void_p(z_host.data_ptr()),
                               ct.c_void_p(c_host.data_ptr()), ct.c_void_p(ws.data_ptr()), ws_bytes, sp),
            "sample_host")
        chk(L.qaoa_gradient_host(a.n, dt_code, ct.c_void_p(psi.data_ptr()), ct.c_void_p(lam.data_ptr()),
                                 ct.byref(desc), gp, bp, a.p, ct.c_void_p(gout.data_ptr()),
                                 g_host.ctypes.data_as(ct.POINTER(ct.c_double)), ct.c_void_p(ws.data_ptr()),
                                 ws_bytes, sp), "gradient_host")

    def barrier():
        if world > 1:
            dist.barrier()

    for _ in range(a.warmup):
        step_device()
    torch.cuda.synchronize()

    # ---- timed device region
    clocks = Clocks(local)
    q.timing_read()
    q.timing_enable(True)
    q.launch_count_reset()
    barrier()
    torch.cuda.synchronize()
    clocks.start()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(a.steps):
        step_device()
    ev1.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    barrier()
    launches = q.launch_count()
    q.timing_enable(False)
    kms, kla, kby, dropped = q.timing_read()
    ms = reduce_max(ev0.elapsed_time(ev1), dev)
    step_ms = ms / a.steps
    layers_per_step = 3 * a.p
    value = job_throughput(layers_per_step * a.steps, world, ms / 1e3)

    # ---- end-to-end region (host buffers through the C ABI)
    for _ in range(1):
        step_e2e()
    barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(a.steps):
        step_e2e()
    torch.cuda.synchronize()
    e2e_s = reduce_max(time.perf_counter() - t0, dev)
    e2e_value = job_throughput(layers_per_step * a.steps, world, e2e_s)
    h2d = e.nbytes + (w.nbytes if w is not None else 0) + gam.nbytes + bet.nbytes
    d2h = 16 + shots * 16 + (2 * a.p + 2) * 8

    # ---- secondary measurements (outside the timed step): gradient rate, batched vs plain
    grad = measure_gradient(q, gradient_once, max(1, min(a.steps, 3)))
    batched = None if a.no_batched else measure_batched(q, dev, "c128", a.batch_graphs)
    ttr = None if a.no_ttr else measure_time_to_ratio(q, dev, "c128")

    # ---- roofline of the dominant kernel (layer sweeps), measured live
    peak, peak_kind = measured_peak_hbm()
    sweep_ms, sweep_n, sweep_bytes = kms[0], kla[0], kby[0]
    achieved = (sweep_bytes / (sweep_ms / 1e3)) / 1e9 if sweep_ms > 0 else 0.0
    tr = traffic_record(sweep_source_hash(), f"{a.dtype}_n{a.n}")
    traffic = None
    if tr is not None:
        traffic = tr.get("bytes_per_launch")
    # the method's least HBM traffic for the step's 3p layers: a forward layer reads and
    # writes psi once and reads C, (2S + c) bytes per amplitude; an adjoint layer does so for psi
    # and lambda, 4S + c (S, c: bytes per amplitude and per cost entry); a cut is symmetric under
    # flipping every qubit, so 2^(n - 1) amplitudes carry the state
    S_b = 16 if a.dtype == "c128" else 8
    c_b = 4 if integer else 8
    min_bytes = float(2 ** (a.n - 1)) * (2 * a.p * (2 * S_b + c_b) + a.p * (4 * S_b + c_b))
    min_gbs = min_bytes / (step_ms / 1e3) / 1e9

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "layers/s", "n_gpus": world, "steps": a.steps,
            "warmup": a.warmup, "ms_per_step": step_ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": arith_dtype(a.dtype), "data": "synthetic",
            "config": {"workload": workload_name(a), "n": a.n, "p": a.p, "state_dtype": a.dtype,
                       "arithmetic": ARITHMETIC[a.dtype],
                       "family": a.family, "weights": a.weights, "shots": shots,
                       "layers_per_step": layers_per_step, "parallelism": f"replicas x{world}",
                       "l2": "inputs larger than L2 (state %.1f GB)" % ((16 if a.dtype == 'c128' else 8) * 2 ** a.n / 1e9)},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "traffic": traffic,
                         "kernel": "layer sweep", "launches": sweep_n,
                         "algorithmic_bytes_per_launch": sweep_bytes / max(1, sweep_n),
                         "peak_source": f"{peak_kind} hbm_gbs",
                         "layer_min_bytes_per_step": min_bytes, "layer_min_gbs": min_gbs,
                         "layer_min_frac": min_gbs / peak},
            "kernels_ms": {"sweep": kms[0], "cost": kms[1], "sample": kms[2], "other": kms[3]},
            "kernels_launches": {"sweep": kla[0], "cost": kla[1], "sample": kla[2], "other": kla[3]},
            "gpu_launches": launches,
            "e2e": {"value": e2e_value, "unit": "layers/s", "h2d_bytes_per_step": int(h2d),
                    "d2h_bytes_per_step": int(d2h)},
            "clocks": clk,
            "gradient": {"workload": f"adjoint gradient (cost vector + forward + adjoint pass), n={a.n}, p={a.p}",
                         **grad},
        }
        if batched is not None:
            line["batched"] = batched
        if ttr is not None:
            line["time_to_ratio"] = ttr
        if not a.no_cpu_baseline:
            line["cpu_baseline"] = cpu_baseline(a)
        emit(line, a)
    if world > 1:
        dist.destroy_process_group()
    return 0


def run_batched(a):
    """The batched workload alone: one JSON line, graph gradients per second."""
    import torch
    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    import paper_2407_13012_gb300 as q
    dev = torch.device("cuda", local)
    res = measure_batched(q, dev, a.dtype, a.batch_graphs, reps=a.steps, autotune=not a.no_autotune)
    if rank == 0:
        emit({"metric": "batched adjoint gradients (graph gradients/s)", "value": res["graph_grads_per_s"],
              "unit": "graph gradients/s", "n_gpus": 1, "steps": a.steps, "warmup": 1,
              "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
              "dtype": arith_dtype(a.dtype), "data": "synthetic",
              "config": {"workload": res["workload"], "arithmetic": ARITHMETIC[a.dtype]}, "batched": res}, a)
    return 0


def run_ttr(a):
    """The time-to-ratio comparison alone: one JSON line, milliseconds for the batched
    optimiser from proposer starts to bring every graph to the target ratio."""
    import torch
    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    import paper_2407_13012_gb300 as q
    dev = torch.device("cuda", local)
    res = measure_time_to_ratio(q, dev, a.dtype, a.ttr_graphs, a.ttr_target)
    if rank == 0:
        emit({"metric": "time to approximation ratio (batched + proposer)",
              "value": res["batched"]["proposer"]["ms_to_ratio"], "unit": "ms", "n_gpus": 1, "steps": 1,
              "warmup": 1, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
              "dtype": arith_dtype(a.dtype), "data": "synthetic",
              "config": {"workload": res["workload"], "arithmetic": ARITHMETIC[a.dtype]}, "time_to_ratio": res}, a)
    return 0


def xy_cpu_baseline(n_small: int = 20, reps: int = 2):
    """The oracle (full 2^n vectors, as it stands) on one layer at n = 20, k = 10, timed on
    the host; returns seconds per layer and the amplitudes it carries."""
    from oracle import qaoa as oq
    from oracle import xy as ox
    import synth
    e, w, _ = synth.graph("reg3", n_small, 0, weights="int")
    C = oq.cut_values(n_small, e, w)
    psi = ox.dicke_state(n_small, n_small // 2)
    t0 = time.perf_counter()
    for _ in range(reps):
        ox.xy_state(n_small, n_small // 2, C, [0.3], [0.4], psi0=psi)
    return (time.perf_counter() - t0) / reps, 1 << n_small


def run_xy(a):
    """QAOA on F_k = {z : popcount(z) = k} with the ring XY mixer: one JSON line, layers/s."""
    import torch
    from math import comb
    import synth
    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    import paper_2407_13012_gb300 as q
    n = a.n
    k = a.k if a.k is not None else n // 2
    fam = "gnp" if (a.family == "reg3" and n % 2) else a.family
    e, w, integer = synth.graph(fam, n, a.seed, weights=a.weights, prob=a.prob)
    g = q.Graph(n, e, w, integer)
    cv = q.xy_cost_vector(g, k, "i32" if integer else "f64")
    gam, bet = synth.angles(a.p, a.seed)
    psi = q.xy_new_state(n, k, a.dtype)
    D = comb(n, k)

    def step():
        return q.xy_apply_layers(psi, n, k, cv, gam, bet, init=True, expect=True)

    for _ in range(a.warmup):
        step()
    torch.cuda.synchronize()
    q.timing_enable(True)
    q.timing_read()
    q.launch_count_reset()
    clocks = Clocks(local)
    clocks.start()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(a.steps):
        out = step()
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / a.steps
    clk = clocks.stop()
    kms, kla, kby, _ = q.timing_read()
    q.timing_enable(False)
    launches = q.launch_count()
    E, nrm = out.cpu().numpy().tolist()
    # the subspace adjoint gradient (forward layers, lambda, backward pass over both buffers)
    lam = q.xy_new_state(n, k, a.dtype)
    q.xy_gradient(psi, lam, n, k, cv, gam, bet)
    torch.cuda.synchronize()
    g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    g0.record()
    for _ in range(max(1, min(a.steps, 3))):
        q.xy_gradient(psi, lam, n, k, cv, gam, bet)
    g1.record()
    torch.cuda.synchronize()
    grad_ms = g0.elapsed_time(g1) / max(1, min(a.steps, 3))
    del lam
    peak, src = measured_peak_hbm()
    achieved = kby[0] / (kms[0] * 1e-3) / 1e9 if kms[0] > 0 else None
    line = {"metric": "xy-mixer QAOA layers per second (Hamming-weight subspace)", "value": a.p * 1e3 / ms,
            "unit": "layers/s", "n_gpus": 1, "steps": a.steps, "warmup": a.warmup, "ms_per_step": ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "int64" if a.dtype == "c128" else "f32", "data": "synthetic",
            "config": {"workload": f"balanced-cut QAOA on F_k: n={n} {'random 3-regular' if fam == 'reg3' else fam}, "
                                   f"k={k} ({D} amplitudes), p={a.p}, ring XY mixer, {a.dtype} subspace state; "
                                   f"step = Dicke start + p layers + <C>", "n": n, "k": k, "p": a.p,
                       "arithmetic": ("float64 pairs in memory; cost unitary and window gate passes (forward and "
                                      "adjoint) in int64 fixed point with a per-tile scale (value = integer x "
                                      "2^-(56 - E), components below 2^E); closing pair and <C> in float64")
                                     if a.dtype == "c128" else
                                     "float32 state and rotations; <C> in float32 chunks summed in float64",
                       "state_dtype": a.dtype, "l2": "state larger than L2, no flush"},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak if achieved else None, "traffic": None,
                         "kernel": "window passes (cost unitary + pair gates) + closing-pair pass", "launches": kla[0],
                         "peak_source": f"{src} hbm_gbs"},
            "gpu_launches": launches, "result": {"E": E, "norm": nrm}, "clocks": clk,
            "gradient": {"workload": f"subspace adjoint gradient, n={n}, k={k}, p={a.p}", "evals_per_s": 1e3 / grad_ms,
                         "ms": grad_ms}}
    if not a.no_cpu_baseline:
        sec, amps = xy_cpu_baseline()
        scale = D / amps * (n / 20)
        line["cpu_baseline"] = {"value": 1.0 / (sec * scale), "unit": "layers/s", "cores": 1, "kind": "oracle",
                                "sample": f"oracle (full 2^20 vectors) on one n=20, k=10 layer, {sec:.2f} s, scaled "
                                          f"by amplitudes and pair gates (x{scale:.0f}) to one layer of this workload"}
    if rank == 0:
        emit(line, a)
    return 0


def main():
    a = parse()
    if a.workload == "xy" and a.impl != "reference":
        return run_xy(a)
    if a.impl == "reference":
        return run_reference(a)
    if a.workload == "batched":
        return run_batched(a)
    if a.workload == "ttr":
        return run_ttr(a)
    return run_ours(a)


if __name__ == "__main__":
    sys.exit(main())
