"""Performance cases of the Graph-VQE engine: what its users have it compute, through its public entry points.

Sizes are those of the workloads in paper_2607_02749_gb300/workloads.py and of the benchmark, or lie between
them: registers of 10 to 30 qubits, 1 to 6 repetitions, every entangler, both precisions, RY and RY+RZ layers,
diagonal and X/Y Hamiltonians, energies alone, energies with gradients, parameter shift, the restricted-update
batch and the readout.

Parameters.  A program that asks for FP64 keeps its angles, energies and gradients in float64.  One that asks for
FP32 amplitudes (the default mode) keeps them in float32, as torch parameters are, and hands them over as the
float64 the calls take; what comes back is kept in float32, the precision that mode computes in.

Each case has a "kind":
  energy   energies of a batch of angle vectors (gradient-free optimisers, line searches)
  grad     energies and adjoint gradients of a batch, some with active-parameter masks
  shift    the parameter-shift gradient
  autograd one training step's forward and backward through the torch autograd function
  batch    many restricted-update problems of different sizes at once
  readout  most probable bitstring, shots and CVaR of the prepared state
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2607_02749_gb300 as gv

LINEAR, CIRCULAR, FULL, REVERSE, PAIRWISE, SCA = range(6)


def listed():
    return [
        # a peptide of the size the method is reported on (8-10 qubits, 4 repetitions, circular): one optimiser
        # step, all latency
        dict(name="peptide_n10_fp64", kind="grad", n=10, reps=4, ent=CIRCULAR, gates=1, batch=1, terms=120, xy=0, fp64=1, mask=0),
        # the small exact workload: 64 candidate vectors at once
        dict(name="energies_n12_fp64", kind="energy", n=12, reps=2, ent=LINEAR, gates=1, batch=64, terms=200, xy=0, fp64=1, mask=0),
        # ... and its parameter-shift gradient (73 energies behind one call)
        dict(name="shift_n12_fp64", kind="shift", n=12, reps=2, ent=LINEAR, gates=1, batch=1, terms=200, xy=0, fp64=1, mask=0),
        # restricted block updates on a mid-size register, circular entangler, odd sizes
        dict(name="blocks_n19_circular", kind="grad", n=19, reps=3, ent=CIRCULAR, gates=1, batch=5, terms=1900, xy=0, fp64=0, mask=1),
        # FP64 refinement of block updates on a register that no longer fits on chip
        dict(name="refine_n21_fp64", kind="grad", n=21, reps=4, ent=LINEAR, gates=1, batch=3, terms=2000, xy=0, fp64=1, mask=1),
        # 256 restricted-update problems of 14-20 qubits and 2-4 repetitions, each with its own Hamiltonian
        dict(name="cluster_256", kind="batch", instances=256, n_lo=14, n_hi=20, reps_lo=2, reps_hi=4, per_qubit=100, fp64=0),
        # global refinement of 16 vectors
        dict(name="refine_n24", kind="grad", n=24, reps=4, ent=LINEAR, gates=1, batch=16, terms=2000, xy=0, fp64=0, mask=0),
        # a gradient-free optimiser's population on the reported circuit (circular, 4 repetitions)
        dict(name="energies_n26_circular", kind="energy", n=26, reps=4, ent=CIRCULAR, gates=1, batch=8, terms=2000, xy=0, fp64=0, mask=0),
        # the full EfficientSU2 layer (RY then RZ) at its usual 3 repetitions and reverse-linear entangler
        dict(name="su2_n24", kind="grad", n=24, reps=3, ent=REVERSE, gates=2, batch=2, terms=2000, xy=0, fp64=0, mask=0),
        # reading out a prepared state: 8192 shots, CVaR 0.2
        dict(name="readout_n26", kind="readout", n=26, reps=4, ent=LINEAR, gates=1, terms=2000, shots=8192, fp64=0),
        # a non-diagonal Hamiltonian trained through autograd
        dict(name="pauli_n28_autograd", kind="autograd", n=28, reps=5, ent=LINEAR, gates=1, batch=2, terms=5000, xy=1, fp64=0, mask=0),
        # the largest register, the benchmark's circuit and Hamiltonian
        dict(name="grad_n30", kind="grad", n=30, reps=6, ent=LINEAR, gates=1, batch=1, terms=20000, xy=0, fp64=0, mask=0),
    ]


def draw(rng):
    """One more case of the same ranges: a work profile, then sizes spread over it."""
    what = rng.choice(["small", "small_energy", "shift", "mid", "mid64", "batch", "many", "energy", "su2", "readout", "xy", "large"])
    ent = rng.choice([LINEAR, LINEAR, CIRCULAR, CIRCULAR, FULL, REVERSE, PAIRWISE, SCA])
    c = dict(kind="grad", reps=rng.randint(1, 5), ent=ent, gates=1, batch=1, xy=0, fp64=0, mask=rng.randint(0, 1))

    def terms(n):
        return int(round(math.exp(rng.uniform(math.log(10 * n), math.log(200 * n)))))

    def fit(n, amps):  # vectors of one call, bounded by the amplitudes they make together
        most = max(1, min(32, int(amps) >> n))
        return int(round(math.exp(rng.uniform(0, math.log(most))))) if most > 1 else 1

    if what == "small":
        n = rng.randint(8, 13)
        c.update(n=n, batch=rng.randint(1, 6), fp64=rng.randint(0, 1))
    elif what == "small_energy":
        n = rng.randint(8, 14)
        c.update(kind="energy", n=n, batch=rng.randint(16, 96), fp64=1, mask=0)
    elif what == "shift":
        n = rng.randint(8, 13)
        c.update(kind="shift", n=n, reps=rng.randint(1, 3), fp64=1)
    elif what == "mid":
        n = rng.randint(14, 21)
        c.update(n=n, batch=fit(n, 1 << 23))
    elif what == "mid64":
        n = rng.randint(14, 22)
        c.update(n=n, batch=fit(n, 1 << 22), fp64=1)
    elif what == "batch":
        lo = rng.randint(14, 16)
        return dict(kind="batch", instances=rng.randint(24, 200), n_lo=lo, n_hi=rng.randint(lo + 1, 20), reps_lo=rng.randint(1, 2),
                    reps_hi=rng.randint(3, 4), per_qubit=rng.randint(20, 100), fp64=0)
    elif what == "many":
        n = rng.randint(22, 25)
        c.update(n=n, batch=fit(n, 1 << 27))
    elif what == "energy":
        n = rng.randint(20, 27)
        c.update(kind="energy", n=n, reps=rng.randint(2, 6), batch=fit(n, 1 << 28), mask=0)
    elif what == "su2":
        n = rng.randint(14, 25)
        c.update(n=n, gates=2, reps=rng.randint(1, 4), batch=fit(n, 1 << 24))
    elif what == "readout":
        n = rng.randint(14, 27)
        return dict(kind="readout", n=n, reps=c["reps"], ent=ent, gates=1, terms=terms(n), shots=rng.randint(1024, 8192), fp64=0)
    elif what == "xy":
        n = rng.randint(15, 27)
        c.update(kind="autograd", n=n, batch=fit(n, 1 << 27), xy=1, mask=0)
    else:
        n = rng.randint(26, 29)
        c.update(n=n, reps=rng.randint(2, 6))
    c.setdefault("terms", terms(n))
    return c


# ---------------------------------------------------------------- inputs --
def _strings(n, terms, rng, xy):
    """Pauli strings of weight 1..4 on uniform qubits: Z-strings with contact and penalty coefficients (three
    quarters c ~ U(-7.5, -0.1), one quarter +10), or, with xy, c ~ N(0, 1) and X/Y letters on 40% of the strings."""
    letters = np.zeros((terms, n), dtype=np.int64)  # 0..3: I, X, Y, Z
    weight = rng.integers(1, min(4, n) + 1, size=terms)
    place = np.argsort(rng.random((terms, n)), axis=1)[:, :4]
    for k in range(min(4, n)):
        rows = np.nonzero(weight > k)[0]
        letters[rows, place[rows, k]] = 3
    if xy:
        for r in np.nonzero(rng.random(terms) < 0.4)[0]:
            at = np.nonzero(letters[r])[0]
            pick = rng.integers(1, 4, size=at.size)
            if np.all(pick == 3):
                pick[rng.integers(0, at.size)] = rng.integers(1, 3)
            letters[r, at] = pick
        coeffs = rng.standard_normal(terms)
    else:
        coeffs = np.where(np.arange(terms) < round(0.75 * terms), rng.uniform(-7.5, -0.1, size=terms), 10.0)
    return letters, coeffs


def _problem(n, reps, gates, batch, terms, xy, mask, rng):
    letters, coeffs = _strings(n, terms, rng, xy)
    params = gates * n * (reps + 1)
    theta = rng.uniform(-math.pi, math.pi, size=(batch, params))
    active = None
    if mask:  # a block of 30 to 60 percent of the parameters of each vector
        share = rng.uniform(0.3, 0.6, size=(batch, 1))
        active = (rng.random((batch, params)) < share).astype(np.uint8)
        active[:, 0] = 1
    return letters, coeffs, theta, active


def _text(letters):
    rows = np.frombuffer(b"IXYZ", dtype=np.uint8)[letters]
    return [r.tobytes().decode() for r in rows]


def _instances(case, seed):
    sizes = np.random.Generator(np.random.PCG64(1000 + case["instances"]))  # the case's; the values are the seed's
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for _ in range(case["instances"]):
        n = int(sizes.integers(case["n_lo"], case["n_hi"] + 1))
        reps = int(sizes.integers(case["reps_lo"], case["reps_hi"] + 1))
        out.append((n, reps) + _problem(n, reps, 1, 1, case["per_qubit"] * n, 0, 1, rng))
    return out


def _angles(theta, fp64):
    return np.asarray(theta, dtype=np.float64 if fp64 else np.float32)


def _one(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return _problem(case["n"], case["reps"], case["gates"], case.get("batch", 1), case["terms"], case.get("xy", 0),
                    case.get("mask", 0), rng)


def prepare(case, seed):
    kind, fp64 = case["kind"], bool(case["fp64"])
    if kind == "batch":
        insts = _instances(case, seed)
        ans = [gv.Ansatz(i[0], i[1]) for i in insts]
        hams = [gv.Hamiltonian(i[0], _text(i[2]), i[3]) for i in insts]
        sizes = [i[4].size for i in insts]
        theta = torch.as_tensor(_angles(np.concatenate([i[4][0] for i in insts]), fp64), device="cuda")
        work = torch.empty_like(theta, dtype=torch.float64)
        grad = torch.empty_like(work)
        masks = [torch.as_tensor(i[5][0], device="cuda") for i in insts]
        return dict(case=case, batch=gv.Batch(ans, hams, fp64=fp64), theta=theta, work=work, grad=grad, masks=masks,
                    params=list(work.split(sizes)), grads=list(grad.split(sizes)))
    letters, coeffs, theta, active = _one(case, seed)
    a = gv.Ansatz(case["n"], case["reps"], entangler=case["ent"], gates=case["gates"])
    h = gv.Hamiltonian(case["n"], _text(letters), coeffs)
    t = torch.as_tensor(_angles(theta, fp64), device="cuda")
    if kind == "autograd":
        t.requires_grad_(True)
    s = dict(case=case, a=a, h=h, theta=t, mask=None if active is None else torch.as_tensor(active, device="cuda"))
    if kind == "readout":
        u = np.random.Generator(np.random.PCG64(seed + 1)).random(case["shots"])
        s["uniforms"] = torch.as_tensor(u, device="cuda")
    return s


def run(state):
    case = state["case"]
    kind, fp64 = case["kind"], bool(case["fp64"])
    if kind == "batch":
        state["work"].copy_(state["theta"])
        e = state["batch"].run(state["params"], masks=state["masks"], grads=state["grads"])
        return dict(e=e, grad=state["grad"]) if fp64 else dict(e=e.float(), grad=state["grad"].float())
    a, h, theta = state["a"], state["h"], state["theta"]
    if kind == "autograd":
        e = gv.GvqeEnergy.apply(theta.double(), a, h, state["mask"], fp64)
        (g,) = torch.autograd.grad(e.sum(), theta)
        return dict(e=e.detach().to(theta.dtype), grad=g)
    t = theta.double()
    if kind == "energy":
        return dict(e=gv.energy(a, h, t, fp64=fp64).to(theta.dtype))
    if kind == "readout":
        r = gv.readout(a, h, t, alpha=0.2, uniforms=state["uniforms"], fp64=fp64)
        return dict(argmax=r.argmax, p_max=r.p_max, cvar=r.cvar, total=r.total, shots=r.shots)
    e, g = gv.energy_grad(a, h, t, mask=state["mask"], fp64=fp64, param_shift=kind == "shift")
    return dict(e=e.to(theta.dtype), grad=g.to(theta.dtype))


def work(case):
    """Bytes: angles and masks read, results written, and the Hamiltonian: its diagonal 2^n numbers of the
    amplitude's type, once for all vectors of a call, and for the readout also the state once.  Flops: one
    multiply-add per amplitude of the diagonal and its energy and, per gate, none: how a state comes about is
    the path's own affair."""
    size = 8 if case["fp64"] else 4
    if case["kind"] == "batch":
        mean = sum(2.0 ** n for n in range(case["n_lo"], case["n_hi"] + 1)) / (case["n_hi"] - case["n_lo"] + 1)
        amps = case["instances"] * mean
        par = case["instances"] * 0.5 * (case["n_lo"] + case["n_hi"]) * (0.5 * (case["reps_lo"] + case["reps_hi"]) + 1)
        return dict(bytes=amps * size + par * 2 * size, flops=4.0 * amps)
    amps = 2.0 ** case["n"]
    vectors = case.get("batch", 1)
    par = vectors * case["gates"] * case["n"] * (case["reps"] + 1)
    states = 1 + (2 * par if case["kind"] == "shift" else 0)
    return dict(bytes=amps * size * (2 if case["kind"] == "readout" else 1) + 2.0 * par * size,
                flops=4.0 * amps * vectors * case["gates"] * states)


# ----------------------------------------------------- the same in 64 bits --
def _cnots(ent, n, layer):
    ring = [(n - 1, 0)] + [(i, i + 1) for i in range(n - 1)]
    if ent == CIRCULAR:
        return ring
    if ent == FULL:
        return [(i, j) for i in range(n) for j in range(i + 1, n)]
    if ent == REVERSE:
        return [(i, i + 1) for i in range(n - 2, -1, -1)]
    if ent == PAIRWISE:
        return [(i, i + 1) for i in range(0, n - 1, 2)] + [(i, i + 1) for i in range(1, n - 1, 2)]
    if ent == SCA:
        s = (layer - 1) % n
        rot = ring[n - s:] + ring[:n - s]
        return [(t, c) for c, t in rot] if (layer - 1) % 2 else rot
    return ring[1:]


def _sources(ent, n, layer, inverse, dev):
    """Index of the amplitude that each place takes its value from: y -> A^-1 y, or (inverse) x -> A x."""
    gates = _cnots(ent, n, layer)
    idx = torch.zeros(1, dtype=torch.int64, device=dev)
    for q in range(n):
        col = 1 << q
        for c, t in (gates if inverse else reversed(gates)):
            col ^= ((col >> c) & 1) << t
        idx = torch.cat([idx, idx ^ col])
    return idx


def _halves(v, q):
    w = v.view(-1, 2, 1 << q)
    return w[:, 0], w[:, 1]


def _ry(v, q, t):
    c, s = math.cos(0.5 * t), math.sin(0.5 * t)
    a, b = _halves(v, q)
    a0 = torch.mul(a, c).sub_(b, alpha=s)
    b.mul_(c).add_(a, alpha=s)
    a.copy_(a0)


def _rz(v, q, t):
    a, b = _halves(v, q)
    a.mul_(complex(math.cos(0.5 * t), -math.sin(0.5 * t)))
    b.mul_(complex(math.cos(0.5 * t), math.sin(0.5 * t)))


def _dot(a, b):
    return torch.real((a.conj() * b).sum()) if a.is_complex() else (a * b).sum()


def _diagonal(n, letters, coeffs, dev):
    """Every diagonal entry of the I/Z strings: the coefficients at their masks, then a Walsh-Hadamard transform."""
    only = np.all((letters == 0) | (letters == 3), axis=1)
    z = ((letters[only] == 3).astype(np.int64) << np.arange(n)).sum(axis=1)
    table = np.zeros(0) if not only.any() else coeffs[only]
    d = torch.zeros(1 << n, dtype=torch.float64, device=dev)
    d.index_add_(0, torch.as_tensor(z, device=dev), torch.as_tensor(table, device=dev))
    for q in range(n):
        a, b = _halves(d, q)
        t = a - b
        a.add_(b)
        b.copy_(t)
    return d, letters[~only], coeffs[~only]


def _apply_strings(out, psi, n, letters, coeffs):
    """out += sum of the strings with X or Y letters on a real state (an odd number of Y gives nothing real)."""
    for row, c in zip(letters, coeffs):
        ny = int((row == 2).sum())
        if ny % 2:
            continue
        at = [int(q) for q in np.nonzero(row)[0]][::-1]
        dims, last = [], n
        for q in at:
            dims += [1 << (last - q - 1), 2]
            last = q
        dims.append(1 << last)
        axes = {q: 2 * k + 1 for k, q in enumerate(at)}
        sign = torch.full([2 if k % 2 else 1 for k in range(len(dims))], float(c) * (-1.0 if ny % 4 == 2 else 1.0),
                          dtype=torch.float64, device=psi.device)
        for q in at:
            if row[q] != 1:  # a sign on the bit of the source
                shape = [1] * len(dims)
                shape[axes[q]] = 2
                sign = sign * torch.tensor([1.0, -1.0], dtype=torch.float64, device=psi.device).view(shape)
        flips = [axes[q] for q in at if row[q] in (1, 2)]
        # <x|P|psi> takes psi at x with the X and Y bits flipped, with the sign of that source
        out.view(dims).addcmul_(psi.view(dims).flip(flips), sign.flip(flips))


def _run64(n, reps, ent, gates, theta, diag, letters, coeffs, grad):
    dev = diag.device
    psi = torch.zeros(1 << n, dtype=torch.complex128 if gates == 2 else torch.float64, device=dev)
    psi[0] = 1.0
    width = gates * n
    for r in range(reps + 1):
        if r:
            psi = psi[_sources(ent, n, r, False, dev)]
        for q in range(n):
            _ry(psi, q, theta[r * width + q])
        if gates == 2:
            for q in range(n):
                _rz(psi, q, theta[r * width + n + q])
    lam = psi * diag
    _apply_strings(lam, psi, n, letters, coeffs)
    e = _dot(psi, lam)
    if not grad:
        return e, None
    g = [None] * (width * (reps + 1))
    for r in range(reps, -1, -1):
        if gates == 2:
            for q in range(n):  # d RZ = -i/2 Z RZ: dE = Im <lambda|Z|psi>
                (p0, p1), (l0, l1) = _halves(psi, q), _halves(lam, q)
                g[r * width + n + q] = (l0.conj() * p0).imag.sum() - (l1.conj() * p1).imag.sum()
            for q in range(n):
                _rz(psi, q, -theta[r * width + n + q])
                _rz(lam, q, -theta[r * width + n + q])
        for q in range(n):  # d RY = 1/2 [[0, -1], [1, 0]] RY: dE = <lambda_1|psi_0> - <lambda_0|psi_1>
            (p0, p1), (l0, l1) = _halves(psi, q), _halves(lam, q)
            g[r * width + q] = _dot(l1, p0) - _dot(l0, p1)
        if r:
            for q in range(n):
                _ry(psi, q, -theta[r * width + q])
                _ry(lam, q, -theta[r * width + q])
            src = _sources(ent, n, r, True, dev)
            psi, lam = psi[src], lam[src]
            del src
    return e, torch.stack([x.to(torch.float64) for x in g])


def _all64(n, reps, ent, gates, thetas, letters, coeffs, active, grad, dev):
    diag, left, lc = _diagonal(n, letters, coeffs, dev)
    es, gs = [], []
    for b in range(thetas.shape[0]):
        e, g = _run64(n, reps, ent, gates, [float(x) for x in thetas[b]], diag, left, lc, grad)
        es.append(e)
        if grad:
            gs.append(g if active is None else g * torch.as_tensor(active[b], dtype=torch.float64, device=dev))
    return torch.stack(es), torch.stack(gs) if grad else None


def _readout64(case, seed, dev):
    n = case["n"]
    letters, coeffs, theta, _ = _one(case, seed)
    diag, _, _ = _diagonal(n, letters, coeffs, dev)
    t = [float(x) for x in _angles(theta, case["fp64"])[0]]
    psi = torch.zeros(1 << n, dtype=torch.float64, device=dev)
    psi[0] = 1.0
    for r in range(case["reps"] + 1):
        if r:
            psi = psi[_sources(case["ent"], n, r, False, dev)]
        for q in range(n):
            _ry(psi, q, t[r * n + q])
    p = psi * psi
    total = p.sum()
    order = torch.argsort(diag)
    mass = torch.cumsum(p[order] / total, 0)
    before = torch.cat([mass.new_zeros(1), mass[:-1]])
    part = (torch.clamp(mass, max=0.2) - before).clamp_(min=0.0)
    cvar = (part * diag[order]).sum() / 0.2
    return dict(argmax=None, p_max=p.max(), cvar=cvar, total=total, shots=None)


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "batch":
        es, gs = [], []
        for n, reps, letters, coeffs, theta, active in _instances(case, seed):
            e, g = _all64(n, reps, LINEAR, 1, _angles(theta, case["fp64"]), letters, coeffs, active, True, dev)
            es.append(e)
            gs.append(g[0])
        return dict(e=torch.cat(es), grad=torch.cat(gs))
    if case["kind"] == "readout":
        return _readout64(case, seed, dev)
    letters, coeffs, theta, active = _one(case, seed)
    grad = case["kind"] != "energy"
    e, g = _all64(case["n"], case["reps"], case["ent"], case["gates"], _angles(theta, case["fp64"]), letters, coeffs, active,
                  grad, dev)
    return dict(e=e, grad=g) if grad else dict(e=e)
