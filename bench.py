#!/usr/bin/env python3
"""Benchmark of the Graph-VQE energy + adjoint-gradient path on GB300.

Default workload (one GPU): n = 30 qubits, reps = 6 (P = 210 parameters), a
diagonal folding-style Hamiltonian of 20,000 Z-strings (15,000 contact terms
c ~ U(-7.5, -0.1), 5,000 penalty terms c = +10), 4 parameter vectors per
step, FP32 amplitudes with FP64 table and reductions.  One step = one
gvqe_energy_grad call for the 4 vectors (energies and the full adjoint
gradient).  Inputs are synthetic and seeded.

Printed JSON line (rank 0): metric/value/unit (E+grad evaluations per second,
device-timed with CUDA events on the launching stream), e2e (same metric through
the public API with pinned host inputs copied in and results copied out every
step), roofline of the dominant kernel (the contraction of the half tables: TF32
tensor operations / measured launch time vs half the measured bf16 rate; tile passes:
algorithmic bytes vs the measured HBM copy bandwidth), the FP64 parameter-shift comparator
on the same GPU, FP32-vs-FP64 errors, clocks during the timed region and the
CPU oracle baseline.

--impl reference times the CPU oracle (the plain complex128 gate-by-gate
simulator in oracle/) on bounded samples of the same workload instead.

Multi-GPU: one process per GPU (torchrun); each rank evaluates its own 4
parameter vectors (independent units, no data-path collective: weak scaling).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import re
import math
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "E+grad evals/s at n=30: FP32 adjoint vs FP64 param-shift; HBM GB/s vs peak"
UNIT = "E+grad/s"
FALLBACK_HBM_GBS = 6800.0


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gvqe", choices=["gvqe", "reference"])
    ap.add_argument("--workload", default="n30_reps6_z20000")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-comparators", action="store_true", help="skip the FP64 comparator legs")
    ap.add_argument("--only-readout", action="store_true",
                    help="run only the readout leg on the workload and print its JSON object")
    ap.add_argument("--only-entanglers", action="store_true",
                    help="run only the entangler leg on the workload and print its JSON object")
    ap.add_argument("--only-su2", action="store_true",
                    help="run only the EfficientSU2 (RY+RZ, complex) leg on the workload and print its JSON object")
    ap.add_argument("--only-driver", action="store_true",
                    help="run only the Graph-VQE driver leg (one epoch at n=20) and print its JSON object")
    ap.add_argument("--only-xy", action="store_true",
                    help="run only the non-diagonal leg (default n=28, 5,000 mixed strings, 8 vectors; "
                         "--xy-workload picks another) and print its JSON object")
    ap.add_argument("--xy-workload", default="n28_reps5_pauli5000")
    ap.add_argument("--only-configs", action="store_true",
                    help="run only the small named workloads (C1 n=12 FP64, C2 n=24 FP32) and print their JSON object")
    ap.add_argument("--only-cluster", action="store_true",
                    help="run only the 256-instance cluster batch leg and print its JSON object")
    ap.add_argument("--no-tune", action="store_true", help="keep the default tile plan (skip the autotuner)")
    ap.add_argument("--mps-layers", type=int, default=0,
                    help="closed-form leading layers (GVQE_OPT_MPS_LAYERS: 0 auto, -1 none, 1..4)")
    ap.add_argument("--mps-tensor", type=int, default=0,
                    help="bond-16 closed-form gradient pass (GVQE_OPT_MPS_TENSOR: 0 tensor cores, -1 FP32 pipe)")
    ap.add_argument("--cpu-single-core", action="store_true",
                    help="also time one full oracle E+grad at n=24 on one core (about 3-4 minutes)")
    return ap.parse_args()


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def max_over_ranks(value: float, dist, device) -> float:
    """The largest value over all ranks (a timed region's duration), or value itself alone."""
    if dist is None:
        return value
    import torch

    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.item()


def measured_peaks(key="hbm_gbs", fallback=FALLBACK_HBM_GBS):
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            d = json.load(f)
        return float(d[key]), "measured"
    except Exception:
        return fallback, "fallback"


def workload_sweeps(n: int, reps: int, n_terms: int):
    """Full-state sweeps of the plain gate-by-gate oracle for one E+grad."""
    ry = (reps + 1) * n          # forward RY gates
    cx = reps * (n - 1)          # forward CNOTs
    # forward + backward (gradient inner product + two inverse gates per RY, two CNOTs per CNOT)
    gate_sweeps = ry + cx + ry * 3 + cx * 2
    return gate_sweeps, n_terms


def oracle_sample(n: int, reps: int, ham, n_gates: int = 2, n_terms: int = 2, single_thread: bool = False):
    """Time a bounded sample of the oracle on the full-size state and scale to one E+grad."""
    import oracle

    t0 = time.perf_counter()
    t_gate, t_term = oracle.sweep_times(n, n_gates, ham.strings[:n_terms], ham.coeffs[:n_terms])
    sampled = time.perf_counter() - t0
    gs, ts = workload_sweeps(n, reps, ham.n_terms)
    sec = gs * t_gate + ts * t_term
    out = {
        "value": 1.0 / sec,
        "unit": UNIT,
        "cores": oracle.max_threads(),
        "kind": "oracle",
        "extrapolated": True,
        "sampled_s": sampled,
        "sample": (f"oracle complex128 at n={n}: {n_gates} RY sweeps ({t_gate:.3f} s each) and {n_terms} "
                   f"Pauli-term sweeps ({t_term:.3f} s each), timed in {sampled:.1f} s wall and scaled to one "
                   f"E+grad = {gs} gate sweeps + {ts} term sweeps = {sec:.0f} s"),
    }
    if single_thread:  # the plain oracle on one core, same scaling
        threads = oracle.max_threads()
        oracle.set_threads(1)
        try:
            g1, t1 = oracle.sweep_times(n, 1, ham.strings[:1], ham.coeffs[:1])
        finally:
            oracle.set_threads(threads)
        sec1 = gs * g1 + ts * t1
        out["single_thread"] = {"value": 1.0 / sec1, "unit": UNIT, "cores": 1, "extrapolated": True,
                                "sample": f"1 RY sweep ({g1:.3f} s) and 1 Pauli-term sweep ({t1:.3f} s) on one "
                                          f"core, scaled the same way = {sec1:.0f} s"}
    return out


def oracle_measured(workload: str = "n24_reps4_z2000", single_core: bool = False):
    """One whole oracle E+grad (gate-by-gate adjoint) of a named workload, timed
    end to end on all host cores (and on one core when asked): measured, not scaled."""
    import oracle
    from paper_2607_02749_gb300 import workloads as wl

    w = wl.WORKLOADS[workload]
    ham, th = wl.make_workload(workload, batch=1)
    out = {"workload": workload, "unit": UNIT, "kind": "oracle", "extrapolated": False}
    runs = [("all_cores", oracle.max_threads())] + ([("single_core", 1)] if single_core else [])
    threads = oracle.max_threads()
    for name, k in runs:
        oracle.set_threads(k)
        try:
            t0 = time.perf_counter()
            e, _ = oracle.energy_grad(w["n"], w["reps"], th[0], ham.strings, ham.coeffs)
            dt = time.perf_counter() - t0
        finally:
            oracle.set_threads(threads)
        out[name] = {"value": 1.0 / dt, "seconds_per_E+grad": dt, "cores": k, "E": e}
    return out


class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = os.path.join("/tmp", f"gvqe_clocks_{os.getpid()}.csv")

    def start(self):
        try:
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "200",
                 "-i", str(self.gpu)], stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        sm, smax, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax = max(smax, float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": smax, "reasons": sorted(reasons),
                "samples": len(sm)}


def kernel_source_hash() -> str:
    h = hashlib.sha256()
    for f in ("gvqe_tile.cuh", "gvqe_kernels.cu", "gvqe_engine.cuh", "gvqe_grad_l0.cu"):
        with open(os.path.join(ROOT, "paper_2607_02749_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def ncu_traffic(kernel: str, bytes_per_launch_units: float):
    """DRAM bytes per launch from the committed ncu summary, if it matches this kernel source."""
    p = os.path.join(ROOT, "profiles", "ncu_traffic.json")
    try:
        with open(p) as f:
            d = json.load(f)
        e = d.get(kernel)
        if not e or e.get("source_hash") != kernel_source_hash():
            return None
        return e["dram_bytes_per_amplitude"] * bytes_per_launch_units
    except Exception:
        return None


def cluster_leg(steps: int):
    """256 independent restricted-update problems (n ~ U{14..20}, reps ~ U{2..4}, own
    Z-string Hamiltonians and 30-60% active masks) in one persistent launch per run."""
    import torch

    import paper_2607_02749_gb300 as gv
    from paper_2607_02749_gb300 import _lib
    from paper_2607_02749_gb300 import workloads as wl

    insts = wl.cluster_batch(256)
    ans = [gv.Ansatz(i.n_qubits, i.reps) for i in insts]
    hams = [gv.Hamiltonian.from_workload(i.ham) for i in insts]
    b = gv.Batch(ans, hams)
    params = [torch.as_tensor(i.theta[0], dtype=torch.float64, device="cuda") for i in insts]
    masks = [torch.as_tensor(i.mask[0], dtype=torch.uint8, device="cuda") for i in insts]
    grads = [torch.empty_like(p) for p in params]
    energies = torch.empty(len(insts), dtype=torch.float64, device="cuda")
    tune = b.autotune(params, masks=masks, grads=grads, energies=energies)
    for _ in range(3):
        b.run(params, masks=masks, grads=grads, energies=energies)
    torch.cuda.synchronize()
    n0 = _lib.gvqe_launch_count()
    t0 = time.perf_counter()
    for _ in range(steps):
        b.run(params, masks=masks, grads=grads, energies=energies)
    torch.cuda.synchronize()
    dt = (time.perf_counter() - t0) / steps
    launches = (_lib.gvqe_launch_count() - n0) / steps
    # the same instances one gvqe_energy_grad call at a time, for comparison
    e1 = torch.empty(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for k in range(len(insts)):
        _lib.gvqe_energy_grad(ans[k].handle, hams[k].handle, params[k], masks[k], e1, grads[k])
    torch.cuda.synchronize()
    dt_loop = time.perf_counter() - t0
    amps = sum(2 ** i.n_qubits for i in insts)
    return {"value": len(insts) / dt, "unit": "E+grad/s", "instances": len(insts), "ms_per_run": dt * 1e3,
            "launches_per_run": launches, "per_instance_calls_ms": dt_loop * 1e3,
            "total_amplitudes": amps, "schedule": tune.strip().splitlines(),
            "tuned_ms_per_run": _tuned_ms(tune),
            "note": "evaluated from the registers' halves: no state is stored, so there are no bytes of state passes to count",
            "timing": "wall clock around synchronous gvqe_batch_run calls (tuned_ms_per_run: CUDA events)"}


def _tuned_ms(report: str):
    """The chosen schedule's CUDA-event time per run from the batch autotuner's report."""
    import re

    m = re.search(r"([0-9.]+) ms per run", report)
    return float(m.group(1)) if m else None


def readout_leg(n: int, reps: int, ham, steps: int):
    """Readout of the benchmark's state (Section IV-F, Section V-A): most probable
    bitstring, 8192 shots and CVaR at alpha = 0.2, FP32, one parameter vector."""
    import numpy as np
    import torch

    import paper_2607_02749_gb300 as gv
    from paper_2607_02749_gb300 import workloads as wl

    a = gv.Ansatz(n, reps)
    h = gv.Hamiltonian.from_workload(ham)
    th = torch.as_tensor(wl.thetas(n, reps, 1, seed=1)[0], dtype=torch.float64, device="cuda")
    u = torch.as_tensor(np.random.Generator(np.random.PCG64(0)).random(8192), device="cuda")
    r = gv.readout(a, h, th, alpha=0.2, uniforms=u)
    gv.readout(a, None, th, alpha=0.0, shots=0)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(steps):
        r = gv.readout(a, h, th, alpha=0.2, uniforms=u)
    torch.cuda.synchronize()
    t_all = (time.perf_counter() - t0) / steps
    t0 = time.perf_counter()
    for _ in range(steps):
        gv.readout(a, None, th, alpha=0.0, shots=0)
    torch.cuda.synchronize()
    t_state = (time.perf_counter() - t0) / steps
    amps = 2 ** n
    # CVaR search: the FP64 table once for its range, once per histogram pass
    # and once for the tail sums; the amplitudes once for the tail sums
    cvar_bytes = (8 * (r.passes + 2) + 4) * amps
    a.close()
    h.close()
    return {"ms_per_readout": t_all * 1e3, "ms_state_and_argmax": t_state * 1e3,
            "ms_shots_and_cvar": (t_all - t_state) * 1e3, "shots": 8192, "alpha": 0.2,
            "cvar_histogram_passes": r.passes, "cvar_min_bytes": cvar_bytes,
            "cvar_GBps": cvar_bytes / max(t_all - t_state, 1e-9) / 1e9,
            "argmax": r.argmax, "p_max": r.p_max, "cvar": r.cvar, "total": r.total,
            "timing": "wall clock around synchronous gvqe_readout calls (state preparation included)"}


def entangler_leg(n: int, reps: int, ham, steps: int):
    """E+grad/s of the benchmark workload (one vector) with each entangler (Section IV-B, Table 2)."""
    import torch

    import paper_2607_02749_gb300 as gv
    from paper_2607_02749_gb300 import workloads as wl

    h = gv.Hamiltonian.from_workload(ham)
    th = torch.as_tensor(wl.thetas(n, reps, 1, seed=1), dtype=torch.float64, device="cuda")
    out = {}
    for name, ent in (("linear", gv.GVQE_ENT_LINEAR), ("circular", gv.GVQE_ENT_CIRCULAR), ("full", gv.GVQE_ENT_FULL),
                      ("reverse_linear", gv.GVQE_ENT_REVERSE_LINEAR), ("pairwise", gv.GVQE_ENT_PAIRWISE),
                      ("sca", gv.GVQE_ENT_SCA)):
        a = gv.Ansatz(n, reps, entangler=ent)
        e, g = gv.energy_grad(a, h, th)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(steps):
            e, g = gv.energy_grad(a, h, th)
        torch.cuda.synchronize()
        dt = (time.perf_counter() - t0) / steps
        out[name] = {"value": 1.0 / dt, "unit": UNIT, "E": float(e.item())}
        a.close()
    h.close()
    out["timing"] = "wall clock around synchronous single-vector gvqe_energy_grad calls (FP32 adjoint)"
    return out


def su2_leg(n: int, reps: int, ham, steps: int):
    """The full EfficientSU2 rotation layer (RY then RZ on every qubit, Eq. 8) on
    the benchmark workload: complex amplitudes, P = 2 n (D+1), one vector per call.
    Per-kind GB/s from the library's CUDA-event profile over the timed calls."""
    import numpy as np
    import torch

    import paper_2607_02749_gb300 as gv
    from paper_2607_02749_gb300 import _lib

    a = gv.Ansatz(n, reps, gates=gv.GVQE_GATES_RY_RZ)
    h = gv.Hamiltonian.from_workload(ham)
    th = torch.as_tensor(np.random.default_rng(1).uniform(-np.pi, np.pi, (1, a.n_params)), device="cuda")
    tune = a.autotune(h, th, cache=os.environ.get("GVQE_TUNE_CACHE", os.path.join("/tmp", "gvqe_tune.json")))
    e, g = gv.energy_grad(a, h, th)
    torch.cuda.synchronize()
    _lib.gvqe_profile_reset()
    _lib.gvqe_profile_enable(True)
    t0 = time.perf_counter()
    for _ in range(steps):
        e, g = gv.energy_grad(a, h, th)
    torch.cuda.synchronize()
    dt = (time.perf_counter() - t0) / steps
    _lib.gvqe_profile_enable(False)
    prof = {k: _lib.gvqe_profile_read(k) for k in range(2)}
    _lib.gvqe_profile_reset()
    names = {0: "k_fwd", 1: "k_bwd"}
    peak, peak_src = measured_peaks()
    per_kind = {}
    for k in prof:
        if not prof[k]["launches"]:
            continue
        gbps = prof[k]["bytes"] / (prof[k]["ms"] / 1000.0) / 1e9 if prof[k]["ms"] else 0.0
        per_kind[names[k]] = {"launches": prof[k]["launches"], "ms": prof[k]["ms"], "GBps": gbps,
                              "frac": gbps / peak if peak else None}
    out = {"value": 1.0 / dt, "unit": UNIT, "n_params": a.n_params, "E": float(e.item()),
           "plan": tune.strip().splitlines(),
           "amplitudes": "fp32 complex (2^(n+1) reals), fp64 table and reductions",
           "per_kind": per_kind, "peak_GBps": peak, "peak_source": f"{peak_src} (MEASURED_PEAKS.json hbm_gbs)",
           "timing": "wall clock around synchronous single-vector gvqe_energy_grad calls (FP32 adjoint)"}
    a.close()
    h.close()
    return out


def driver_leg(n: int = 20, reps: int = 4, n_terms: int = 2000):
    """One Graph-VQE epoch (Section IV-C to IV-E) on a sequence-local synthetic H:
    Louvain blocks, lock-step block L-BFGS-B with batched GPU evaluations, global
    refinement.  Reports wall time and evaluation throughput inside the loop."""
    from paper_2607_02749_gb300 import workloads as wl
    from paper_2607_02749_gb300.driver import GraphVQE, GraphVQEConfig

    ham = wl.chain_z_hamiltonian(n, n_terms, seed=0)
    cfg = GraphVQEConfig(reps=reps, max_epochs=1, block_maxiter=60, global_maxiter=30)
    g = GraphVQE(ham, cfg)
    th0 = wl.thetas(n, reps, 1, seed=1)[0]
    g.energy(th0)  # plans and workspaces
    t0 = time.perf_counter()
    r = g.run(th0)
    dt = time.perf_counter() - t0
    ev = g.evaluator
    out = {"workload": f"chain_z n={n} reps={reps} terms={n_terms}", "wall_s": dt, "blocks": r["n_blocks"],
           "modularity": r["modularity"], "E_start": r["E_start"], "E": r["E"],
           "evaluations": r["evaluations"], "gpu_calls": ev.calls, "gpu_rows": ev.rows,
           "rows_per_s": ev.rows / dt, "block_batches": getattr(g, "block_batches", None),
           "timing": "wall clock around GraphVQE.run (host L-BFGS-B, H2D/D2H per call included)"}
    ev.close()
    return out


def xy_masks(ham, tile_bits: int = 13):
    """Distinct X-masks of the strings that reach the real-amplitude path (X/Y
    letters, an even number of Y), and their distinct parts above the tile bits."""
    ms = set()
    for st in ham.strings:
        m = 0
        ny = 0
        for q, L in enumerate(st):
            if L in "XY":
                m |= 1 << q
            ny += L == "Y"
        if m and ny % 2 == 0:
            ms.add(m)
    return len(ms), len({m >> tile_bits for m in ms})


def xy_leg(steps: int, workload: str = "n28_reps5_pauli5000"):
    """The non-diagonal workload: n = 28, reps = 5, 5,000 strings over {I,X,Y,Z}
    (X/Y letters on about 40%), 8 vectors per step through the torch.autograd.Function
    (FP32): energies, then the adjoint gradient by backward().  Per-kind device time
    from the library's CUDA-event profile over the timed steps."""
    import torch

    import paper_2607_02749_gb300 as gv
    from paper_2607_02749_gb300 import _lib
    from paper_2607_02749_gb300 import workloads as wl

    w = wl.WORKLOADS[workload]
    n, reps = w["n"], w["reps"]
    ham, th = wl.make_workload(workload)
    B = th.shape[0]
    a = gv.Ansatz(n, reps)
    h = gv.Hamiltonian.from_workload(ham)
    st = h.stats()
    base = torch.as_tensor(th, dtype=torch.float64, device="cuda")
    tune = a.autotune(h, base, cache=os.environ.get("GVQE_TUNE_CACHE", os.path.join("/tmp", "gvqe_tune.json")))

    def step():
        t = base.clone().requires_grad_(True)
        e = gv.GvqeEnergy.apply(t, a, h, None, False)
        e.sum().backward()
        return e, t.grad

    step()
    torch.cuda.synchronize()
    _lib.gvqe_profile_reset()
    _lib.gvqe_profile_enable(True)
    t0 = time.perf_counter()
    for _ in range(steps):
        e, g = step()
    torch.cuda.synchronize()
    dt = (time.perf_counter() - t0) / steps
    _lib.gvqe_profile_enable(False)
    prof = {k: _lib.gvqe_profile_read(k) for k in range(5)}
    _lib.gvqe_profile_reset()
    names = {0: "k_fwd", 1: "k_bwd", 2: "k_grad_l0", 3: "k_lambda_xy", 4: "k_wht"}
    import re

    m = re.search(r"xy_tile_bits=(\d+)", tune) or re.search(r"tile_bits=(\d+)", tune)
    tb_sel = int(m.group(1)) if m else 13  # the X-mask pass's tile bits
    d_all, d_hi = xy_masks(ham, tb_sel)
    S = 4 * 2 ** n
    T = 8 * 2 ** n
    xy = prof[3]
    lam_ms = xy["ms"] / (steps * B) if xy["launches"] else None
    lam_alg = (2 + d_hi) * S + T  # energy and lambda with the X-mask groups (one partner sweep per high part)
    out = {"value": B / dt, "unit": UNIT, "workload": workload, "n_qubits": n, "reps": reps, "batch": B,
           "n_terms": ham.n_terms, "x_masks": d_all, "D_hi": d_hi, "tile_bits": tb_sel,
           "plan": tune.strip().splitlines(),
           "groups": st["groups"], "grouped_terms": st["grouped"], "dropped_odd_y": st["dropped_odd_y"],
           "ms_per_step": dt * 1e3,
           "per_kind_ms_per_step": {names[k]: prof[k]["ms"] / steps for k in prof if prof[k]["launches"]},
           "k_lambda_xy": {"launches_per_vector": xy["launches"] / (steps * B) if xy["launches"] else 0,
                           "ms_per_vector": lam_ms,
                           "algorithmic_bytes_per_vector": lam_alg,
                           "algorithmic_GBps": (lam_alg / (lam_ms / 1e3) / 1e9) if lam_ms else None,
                           "implementation_GBps": (xy["bytes"] / (xy["ms"] / 1e3) / 1e9) if xy["ms"] else None,
                           "bytes_formula": "(2 + D_hi) S + T, S = 4 B x 2^n (real FP32), T = 8 B x 2^n"},
           "E0": float(e[0].item()),
           "timing": "wall clock around GvqeEnergy forward + backward per 8-vector step (FP32 adjoint)"}
    a.close()
    h.close()
    return out


def configs_leg(steps: int):
    """The two small named workloads, on the GPU:
    C1: n = 12, reps = 2, FP64, 200 Z-strings: energies of 64 parameter vectors in one call
        plus the FP64 parameter-shift gradient (Eq. 13) of one vector (2P + 1 = 73 energies);
    C2: n = 24, reps = 4, FP32 adjoint E+grad of 16 vectors (2,000 Z-strings), plan tuned."""
    import torch

    import paper_2607_02749_gb300 as gv
    from paper_2607_02749_gb300 import workloads as wl

    cache = os.environ.get("GVQE_TUNE_CACHE", os.path.join("/tmp", "gvqe_tune.json"))
    out = {}
    # C1
    ham, th = wl.make_workload("n12_reps2_z200", batch=64)
    a = gv.Ansatz(12, 2)
    h = gv.Hamiltonian.from_workload(ham)
    t = torch.as_tensor(th, device="cuda")

    def c1():
        e = gv.energy(a, h, t, fp64=True)
        _, g = gv.energy_grad(a, h, t[:1], fp64=True, param_shift=True)
        return e, g

    for _ in range(3):
        c1()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(steps):
        c1()
    torch.cuda.synchronize()
    dt = (time.perf_counter() - t0) / steps
    P = a.n_params
    out["C1_n12_reps2_z200_fp64"] = {"value": (64 + 2 * P + 1) / dt, "unit": "energy evals/s",
                                     "ms_per_step": dt * 1e3,
                                     "step": f"64 energies + parameter-shift gradient of one vector ({2 * P + 1} energies)",
                                     "timing": "wall clock around synchronous calls (FP64)"}
    a.close()
    h.close()
    # C2
    ham, th = wl.make_workload("n24_reps4_z2000")
    a = gv.Ansatz(24, 4)
    h = gv.Hamiltonian.from_workload(ham)
    t = torch.as_tensor(th, device="cuda")
    tune = a.autotune(h, t, cache=cache)
    res = {}
    for fp64 in (False, True):
        for _ in range(2):
            gv.energy_grad(a, h, t, fp64=fp64)
        torch.cuda.synchronize()
        ev0 = torch.cuda.Event(enable_timing=True)
        ev1 = torch.cuda.Event(enable_timing=True)
        ev0.record()
        for _ in range(steps):
            gv.energy_grad(a, h, t, fp64=fp64)
        ev1.record()
        torch.cuda.synchronize()
        ms = ev0.elapsed_time(ev1) / steps
        res["fp64" if fp64 else "fp32"] = {"value": th.shape[0] / (ms / 1e3), "unit": UNIT, "ms_per_16": ms}
    out["C2_n24_reps4_z2000"] = {"fp32_adjoint": res["fp32"], "fp64_adjoint": res["fp64"],
                                 "plan": tune.strip().splitlines(),
                                 "timing": "CUDA events around 16-vector gvqe_energy_grad calls"}
    a.close()
    h.close()
    return out


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    from paper_2607_02749_gb300 import workloads as wl

    w = wl.WORKLOADS[args.workload]
    ham, _ = wl.make_workload(args.workload, batch=1)
    n, reps = w["n"], w["reps"]
    vals, walls = [], []
    last = None
    for i in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        r = oracle_sample(n, reps, ham, n_gates=1, n_terms=1)
        wall = time.perf_counter() - t0
        if i >= args.warmup:
            vals.append(r["value"])
            walls.append(wall)
            last = r
    value = statistics.median(vals)
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1000.0 * statistics.mean(walls), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "c128", "data": "synthetic",
        "impl": "reference", "extrapolated": True,
        "timing": ("each step times a bounded sample (one RY sweep and one Pauli-term sweep of the oracle on "
                   "the full 2^n state); ms_per_step is that sample's wall time, value the E+grad rate it "
                   "implies for the whole workload"),
        "config": {"workload": args.workload, "n_qubits": n, "reps": reps, "n_terms": w["terms"],
                   "batch": 4, "parallelism": "replicas"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": last["cores"], "kind": "oracle",
                         "extrapolated": True, "sample": "per step: " + last["sample"]},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(out), flush=True)
    return 0


def run_gvqe(args):
    import numpy as np
    import torch

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    dist = None
    if ws > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl")
    import paper_2607_02749_gb300 as gv
    from paper_2607_02749_gb300 import _lib
    from paper_2607_02749_gb300 import workloads as wl

    w = wl.WORKLOADS[args.workload]
    n, reps, B = w["n"], w["reps"], w["batch"]
    ham, _ = wl.make_workload(args.workload, batch=1)
    if args.only_readout:
        if rank == 0:
            print(json.dumps({"workload": args.workload, "readout": readout_leg(n, reps, ham, max(1, args.steps))}),
                  flush=True)
        return 0
    if args.only_su2:
        if rank == 0:
            print(json.dumps({"workload": args.workload, "efficient_su2": su2_leg(n, reps, ham, max(1, args.steps))}),
                  flush=True)
        return 0
    if args.only_driver:
        if rank == 0:
            print(json.dumps({"driver": driver_leg()}), flush=True)
        return 0
    if args.only_xy:
        if rank == 0:
            print(json.dumps({"non_diagonal": xy_leg(max(1, args.steps), args.xy_workload)}), flush=True)
        return 0
    if args.only_configs:
        if rank == 0:
            print(json.dumps({"configs": configs_leg(max(1, args.steps))}), flush=True)
        return 0
    if args.only_cluster:
        if rank == 0:
            print(json.dumps({"cluster_batch": cluster_leg(max(1, args.steps))}), flush=True)
        return 0
    if args.only_entanglers:
        if rank == 0:
            print(json.dumps({"workload": args.workload,
                              "entanglers": entangler_leg(n, reps, ham, max(1, args.steps))}), flush=True)
        return 0
    theta = wl.thetas(n, reps, B, seed=1 + rank)
    P = n * (reps + 1)
    dev = torch.device("cuda", local)
    h = gv.Hamiltonian.from_workload(ham)
    a = gv.Ansatz(n, reps)
    if args.mps_layers:
        a.set_mps_layers(args.mps_layers)
    if args.mps_tensor:
        a.set_mps_tensor(args.mps_tensor)
    th = torch.as_tensor(theta, dtype=torch.float64, device=dev)
    E = torch.empty(B, dtype=torch.float64, device=dev)
    G = torch.empty(B, P, dtype=torch.float64, device=dev)
    stream = torch.cuda.current_stream()

    # the tile plan: measured by the library's autotuner on this workload (cached per key)
    tune_cache = os.environ.get("GVQE_TUNE_CACHE", os.path.join("/tmp", "gvqe_tune.json"))
    t0 = time.perf_counter()
    tune_report = a.autotune(h, th, cache=tune_cache, stream=stream) if not args.no_tune else "not tuned"
    tune_s = time.perf_counter() - t0

    def step():
        _lib.gvqe_energy_grad(a.handle, h.handle, th, None, E, G, _lib.GVQE_FP32, stream)

    for _ in range(max(3, args.warmup)):
        step()
    torch.cuda.synchronize()

    def barrier():
        if dist is not None:
            dist.barrier()

    gpu_index = local
    cvd = os.environ.get("CUDA_VISIBLE_DEVICES")
    if cvd:
        try:
            gpu_index = int(cvd.split(",")[local])
        except ValueError:
            pass
    clocks = ClockSampler(gpu_index)
    _lib.gvqe_profile_reset()
    _lib.gvqe_profile_enable(True)
    n_launch0 = _lib.gvqe_launch_count()
    clocks.start()
    barrier()
    torch.cuda.synchronize()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(args.steps):
        step()
    ev1.record(stream)
    torch.cuda.synchronize()
    barrier()
    clk = clocks.stop()
    _lib.gvqe_profile_enable(False)
    launches = _lib.gvqe_launch_count() - n_launch0
    ms = max_over_ranks(ev0.elapsed_time(ev1), dist, dev)
    units = ws * B * args.steps
    value = units / (ms / 1000.0)

    # Roofline of the dominant kernel kind, measured live over the timed region.
    # Algorithmic bytes per E+grad (one sweep of the state per layer, real FP32
    # amplitudes S = 4 B x 2^n, FP64 table T = 8 B x 2^n): forward S + 2 D S,
    # backward layers D..1 (3 S + T) + 4 S (D - 1), layer 0 2 S; total (6D+2) S + T.
    # Each kind's share over its measured time is its algorithmic GB/s; the
    # implementation's own per-pass bytes (every tile pass reads and writes the
    # whole state) give the per-pass figure beside it.
    prof = {k: _lib.gvqe_profile_read(k) for k in range(12)}
    names = {0: "k_fwd", 1: "k_bwd", 2: "k_grad_l0", 3: "k_lambda_xy", 4: "k_wht", 5: "k_mps_write",
             6: "k_mps_tab", 7: "k_mps_grad", 8: "k_mps_gtree", 9: "k_mps_gred", 10: "k_mps_genv",
             11: "k_cut_contract_tc"}
    dom = max(prof, key=lambda k: prof[k]["ms"])
    pk = prof[dom]
    peak, peak_src = measured_peaks()
    S_b, T_b = 4.0 * 2 ** n, 8.0 * 2 ** n
    evals = B * args.steps  # E+grad evaluations in the timed region (this rank)
    # layers 1..R in closed form: with their gradients taken from lambda_R, k_bwd
    # sweeps layers D..R+1 only, and the closed-form gradient kernels stand in for
    # the backward of layers R..1 and layer 0 (4 R S + 2 S of the algorithmic count)
    m = re.search(r"closed-form layers 1\.\.(\d+) .*their gradients", a.describe())
    R_cf = int(m.group(1)) if m else 0
    alg_share = {0: (1 + 2 * reps) * S_b, 1: (4 * (reps - R_cf) - 1) * S_b + T_b, 2: 2 * S_b}
    alg_step = ((6 * reps + 2) * S_b + T_b) * B
    def kind_alg(k):
        if not prof[k]["ms"] or k not in alg_share:
            return None
        return alg_share[k] * evals / (prof[k]["ms"] / 1000.0) / 1e9
    pass_gbps = pk["bytes"] / (pk["ms"] / 1000.0) / 1e9 if pk["ms"] > 0 else 0.0
    achieved = kind_alg(dom) or 0.0
    launches_dom = max(1, pk["launches"])
    amps_per_launch = 2.0 ** n
    roofline = {
        "bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
        "traffic": ncu_traffic(names[dom], amps_per_launch),
        "kernel": names[dom], "launches": pk["launches"], "avg_launch_ms": pk["ms"] / launches_dom,
        "algorithmic_bytes_per_launch": alg_share.get(dom, 0.0) * evals / launches_dom,
        "bytes_rule": ("algorithmic: (6D+2) S + T per E+grad, one sweep per layer (forward S + 2DS, k_bwd "
                       "(4D-1) S + T, k_grad_l0 2S; with layers 1..R in closed form and their gradients from "
                       "lambda_R, k_bwd's share is (4(D-R)-1) S + T and the closed-form gradient kernels' "
                       "(4R+2) S); S = 4 B x 2^n real FP32 state, T = 8 B x 2^n FP64 table. "
                       "Layer 0 is an analytic product state here, so the forward never writes it and k_grad_l0 "
                       "reads only lambda; the forward's stored states of layers 1..3 are written in closed "
                       "form (k_mps_tab + k_mps_write, write-only) and the rest by k_fwd tile passes, so the "
                       "forward's algorithmic rate is given for the three kinds together (per_kind.forward)"),
        "per_pass": {"achieved": pass_gbps, "frac": pass_gbps / peak,
                     "bytes_per_launch": pk["bytes"] / launches_dom,
                     "rule": "every tile pass reads and writes the whole state (3 passes per layer at n=30)"},
        "step": {"algorithmic_bytes": alg_step, "achieved": alg_step * args.steps / (ms / 1000.0) / 1e9,
                 "frac": alg_step * args.steps / (ms / 1000.0) / 1e9 / peak},
        "peak_source": f"{peak_src} (MEASURED_PEAKS.json hbm_gbs)" if peak_src == "measured" else "fallback",
        "per_kind": {names[k]: {"launches": prof[k]["launches"], "ms": prof[k]["ms"],
                                "GBps_per_pass": (prof[k]["bytes"] / (prof[k]["ms"] / 1000.0) / 1e9)
                                if prof[k]["ms"] else 0.0,
                                "GBps_algorithmic": kind_alg(k) if k != 0 else None}
                     for k in prof if prof[k]["launches"]},
    }
    fwd_ms = sum(prof[k]["ms"] for k in (0, 5, 6))
    cut = re.search(r"evaluated from the halves .* (\d+) terms", a.describe())
    if dom == 11 and cut:
        # no state is stored: per E+grad S and G once for either half, 2 D 2^n multiply-adds each
        # way, every product as three TF32 ones
        D = int(cut.group(1))
        tf = 24.0 * max(16, D) * 2.0 ** n * evals / (pk["ms"] / 1000.0) / 1e12
        bf16 = measured_peaks("bf16_tflops", 1900.0)
        roofline = {
            "bound": "tensor", "achieved": tf, "peak": bf16[0] / 2, "unit": "TFLOP/s", "frac": tf / (bf16[0] / 2),
            "traffic": None, "kernel": names[dom], "launches": pk["launches"], "avg_launch_ms": pk["ms"] / launches_dom,
            "algorithmic_flops_per_launch": 6.0 * D * 2.0 ** n * evals / launches_dom,
            "tf32_flops_per_launch": 24.0 * max(16, D) * 2.0 ** n * evals / launches_dom,
            "flops_rule": "TF32: S = A B^T (formed for either half) and G = lambda B, 3 products each (hi/lo split), 2 K 2^n "
                          "operations a product; algorithmic: S once and G for either half in one product each",
            "terms": D, "share_of_step": pk["ms"] / ms,
            "table_GBps": pk["bytes"] / (pk["ms"] / 1000.0) / 1e9,
            "peak_source": f"{bf16[1]} (half of MEASURED_PEAKS.json bf16_tflops)" if bf16[1] == "measured" else "fallback",
            "per_kind": {names[k]: {"launches": prof[k]["launches"], "ms": prof[k]["ms"]} for k in prof if prof[k]["launches"]},
        }
    if fwd_ms > 0 and dom != 11:
        roofline["per_kind"]["forward"] = {
            "kinds": "k_fwd + k_mps_write + k_mps_tab", "ms": fwd_ms,
            "GBps_algorithmic": alg_share[0] * evals / (fwd_ms / 1000.0) / 1e9}
    cfg_ms = sum(prof[k]["ms"] for k in (7, 8, 9, 10))
    if R_cf and cfg_ms > 0:
        roofline["per_kind"]["closed_form_gradients"] = {
            "kinds": "k_mps_grad + k_mps_gtree + k_mps_gred + k_mps_genv", "ms": cfg_ms, "layers": R_cf,
            "GBps_algorithmic": (4 * R_cf + 2) * S_b * evals / (cfg_ms / 1000.0) / 1e9,
            "rule": "stand-in for the backward of layers R..1 and layer 0: (4R + 2) S of the algorithmic count"}
    _lib.gvqe_profile_reset()

    # e2e through the public API: pinned host inputs in, results out, every step
    th_host = torch.as_tensor(theta, dtype=torch.float64).pin_memory()
    e_host = torch.empty(B, dtype=torch.float64).pin_memory()
    g_host = torch.empty(B, P, dtype=torch.float64).pin_memory()
    for _ in range(2):
        e_d, g_d = gv.energy_grad(a, h, th_host.to(dev, non_blocking=True))
    torch.cuda.synchronize()
    barrier()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        e_d, g_d = gv.energy_grad(a, h, th_host.to(dev, non_blocking=True))
        e_host.copy_(e_d, non_blocking=True)
        g_host.copy_(g_d, non_blocking=True)
        torch.cuda.current_stream().synchronize()
    e2e_s = max_over_ranks(time.perf_counter() - t0, dist, dev)
    e2e = {"value": ws * B * args.steps / e2e_s, "unit": UNIT, "h2d_bytes_per_step": B * P * 8,
           "d2h_bytes_per_step": B * 8 + B * P * 8}

    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
        "warmup": max(3, args.warmup), "ms_per_step": ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": args.workload, "n_qubits": n, "reps": reps, "n_params": P,
                   "n_terms": w["terms"], "batch_per_gpu": B, "global_batch": B * ws,
                   "amplitudes": "fp32 (real: RY+CX keeps the state real), fp64 table and reductions",
                   "l2": "inputs larger than L2 (two 4 GiB tables per evaluation)", "parallelism": f"replicas x{ws}"},
        "e2e": e2e, "gpu_launches": launches, "roofline": roofline, "clocks": clk,
        "plan": {"autotune": tune_report.strip().splitlines(), "tune_seconds": tune_s, "cache": tune_cache,
                 "layer_passes": [ln.strip() for ln in a.describe().splitlines() if "layer pass" in ln]},
    }

    if rank == 0 and not args.no_comparators:
        # FP32 vs FP64 mode on vector 0, and the FP64 parameter-shift comparator (Eq. 13)
        e32, g32 = E[0].item(), G[0].cpu().numpy()
        t0 = time.perf_counter()
        e64, g64 = gv.energy_grad(a, h, th[:1], fp64=True)
        torch.cuda.synchronize()
        t_adj64 = time.perf_counter() - t0
        e64, g64 = e64.item(), g64[0].cpu().numpy()
        scale = ham.abs_sum()
        out["errors_vs_fp64"] = {"dE_over_sum_abs_c": abs(e32 - e64) / scale,
                                 "grad_rel_l2": float(np.linalg.norm(g32 - g64) / np.linalg.norm(g64)),
                                 "sum_abs_c": scale, "E_fp64": e64}
        mask = torch.zeros(1, P, dtype=torch.uint8, device=dev)
        mask[0, P - 1] = 1
        gv.energy_grad(a, h, th[:1], mask=mask, fp64=True, param_shift=True)  # warm the path
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        _, gps = gv.energy_grad(a, h, th[:1], mask=mask, fp64=True, param_shift=True)
        torch.cuda.synchronize()
        t_3 = time.perf_counter() - t0
        t_grad = t_3 * (2 * P + 1) / 3.0
        out["fp64_param_shift"] = {
            "value": 1.0 / t_grad, "unit": UNIT, "extrapolated": True, "sampled_s": t_3,
            "sample": f"3 FP64 energies (1 active parameter) took {t_3:.3f} s; one gradient = {2 * P + 1} energies",
            "fp64_adjoint_value": 1.0 / t_adj64,
            "check_dE_dtheta_last": {"param_shift": float(gps[0, P - 1].item()), "adjoint_fp64": float(g64[P - 1])},
        }
        out["speedup_fp32_adjoint_vs_fp64_param_shift"] = value / ws / (1.0 / t_grad)

    if rank == 0 and not args.no_comparators:
        a.close()  # the legs below allocate their own workspaces
        out["cluster_batch"] = cluster_leg(args.steps)
        out["readout"] = readout_leg(n, reps, ham, max(1, min(args.steps, 3)))
        out["entanglers"] = entangler_leg(n, reps, ham, max(1, min(args.steps, 3)))
        out["driver"] = driver_leg()
        out["efficient_su2"] = su2_leg(n, reps, ham, max(1, min(args.steps, 3)))
        out["non_diagonal"] = xy_leg(max(1, min(args.steps, 3)))
        out["configs"] = configs_leg(max(1, min(args.steps, 3)))

    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        try:
            out["cpu_baseline"] = oracle_sample(n, reps, ham, single_thread=True)
        except Exception as exc:  # pragma: no cover - host out of memory
            out["cpu_baseline"] = {"value": None, "unit": UNIT, "cores": None, "kind": "oracle",
                                   "sample": f"failed: {exc}"}
        try:
            out["cpu_measured"] = oracle_measured(single_core=args.cpu_single_core)
        except Exception as exc:  # pragma: no cover
            out["cpu_measured"] = {"failed": str(exc)}
    if rank == 0:
        print(json.dumps(out), flush=True)
    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()
    return 0


def main():
    args = parse_args()
    if args.impl == "reference":
        return run_reference(args)
    return run_gvqe(args)


if __name__ == "__main__":
    sys.exit(main())
