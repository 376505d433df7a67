"""The two-half evaluation (gvqe_cut.cuh) against the oracle and the tile passes.

A diagonal H with RY layers whose entanglers cross the middle of the register at
most six times in all is evaluated from two half-register tables instead of a
2^n state.  Sizes: the smallest registers of each precision, odd ones (uneven
halves), every number of terms (2 to 64), every entangler, several row blocks and
column splits, many vectors per launch, masks.  Tolerances as in
test_gpu_parity.py, and against the tile passes of the same precision the FP32
level of both (a few units of 2^-22 per product, averaged over the sums: 5e-6
relative L2 leaves a factor of ten) and 1e-12 in FP64.
"""
import numpy as np
import pytest

import oracle
from paper_2607_02749_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2607_02749_gb300 as gv  # noqa: E402

ALL = [gv.GVQE_ENT_LINEAR, gv.GVQE_ENT_CIRCULAR, gv.GVQE_ENT_FULL, gv.GVQE_ENT_REVERSE_LINEAR, gv.GVQE_ENT_PAIRWISE,
       gv.GVQE_ENT_SCA]
TWO = (gv.GVQE_ENT_CIRCULAR, gv.GVQE_ENT_SCA)  # two crossings per layer


def _run(n, reps, ent, ham, th, fp64, mps=0, mask=None):
    a = gv.Ansatz(n, reps, entangler=ent)
    a.set_mps_layers(mps)
    h = gv.Hamiltonian.from_workload(ham)
    t = torch.as_tensor(th, device="cuda")
    m = None if mask is None else torch.as_tensor(mask, dtype=torch.uint8, device="cuda")
    e0 = gv.energy(a, h, t, fp64=fp64).cpu().numpy()
    e, g = gv.energy_grad(a, h, t, mask=m, fp64=fp64)
    d = a.describe(fp64=fp64)
    a.close()
    h.close()
    return e0, e.cpu().numpy(), g.cpu().numpy(), d


CASES = [(n, r, e, fp64) for e in ALL
         for n, r, fp64 in [(14, 1, False), (15, 3, False), (17, 2, False), (16, 6, False), (18, 5, False),
                            (10, 2, True), (11, 1, True), (12, 3, True), (13, 2, True), (15, 6, True)]
         if not (e in TWO and r > 3)]


@pytest.mark.parametrize("n,reps,ent,fp64", CASES)
def test_against_oracle_and_tile_passes(n, reps, ent, fp64):
    ham = wl.z_hamiltonian(n, 5 * n + 3, seed=n + reps)
    th = wl.thetas(n, reps, 2, seed=10 * n + ent)
    e0, e, g, d = _run(n, reps, ent, ham, th, fp64)
    kappa = (2 if ent in TWO else 1) * reps
    if not fp64:
        assert f"{2 ** kappa} terms" in d, d
    scale = ham.abs_sum()
    te, tg = (1e-10, 1e-9) if fp64 else (2e-5, 1e-4)
    b = 1
    with oracle.entangler(ent):
        er, gr = oracle.energy_grad(n, reps, th[b], ham.strings, ham.coeffs)
    assert abs(e[b] - er) <= te * scale and abs(e0[b] - er) <= te * scale
    if fp64:
        assert np.max(np.abs(g[b] - gr)) <= tg * scale
    else:
        assert np.linalg.norm(g[b] - gr) <= tg * np.linalg.norm(gr)
    _, et, gt, dt = _run(n, reps, ent, ham, th, fp64, mps=-1)
    assert "terms" not in dt
    rel = np.linalg.norm(g - gt) / np.linalg.norm(gt)
    print(f"n={n} reps={reps} ent={ent} fp64={fp64}: oracle grad {np.linalg.norm(g[b] - gr) / np.linalg.norm(gr):.2e} "
          f"(tile passes {np.linalg.norm(gt[b] - gr) / np.linalg.norm(gr):.2e}), E {abs(e[b] - er) / scale:.1e} "
          f"({abs(et[b] - er) / scale:.1e})")
    assert rel <= (1e-12 if fp64 else 5e-6), rel


@pytest.mark.parametrize("n,reps,ent,batch,fp64", [(22, 4, gv.GVQE_ENT_LINEAR, 3, False), (25, 6, gv.GVQE_ENT_FULL, 2, False),
                                                   (24, 2, gv.GVQE_ENT_CIRCULAR, 5, False), (20, 3, gv.GVQE_ENT_PAIRWISE, 2, True)])
def test_many_items_and_vectors(n, reps, ent, batch, fp64):
    """Several row blocks and column splits, E and its transposed copy at unequal
    halves, more items than multiprocessors, masks; single vectors give the same bits."""
    ham = wl.z_hamiltonian(n, 200, seed=n)
    th = wl.thetas(n, reps, batch, seed=n + 1)
    mask = wl.active_mask(n * (reps + 1), batch, seed=n + 2)
    e0, e, g, d = _run(n, reps, ent, ham, th, fp64, mask=mask)
    assert "terms" in d
    _, et, gt, _ = _run(n, reps, ent, ham, th, fp64, mps=-1, mask=mask)
    assert np.all(g[mask == 0] == 0.0)
    scale = ham.abs_sum()
    assert np.max(np.abs(e - et)) <= (1e-12 if fp64 else 1e-7) * scale
    assert np.max(np.abs(e0 - et)) <= (1e-12 if fp64 else 1e-7) * scale
    rel = np.linalg.norm(g - gt) / np.linalg.norm(gt)
    print(f"n={n} reps={reps} ent={ent}: vs tile passes grad {rel:.2e}, E {np.max(np.abs(e - et)) / scale:.1e}")
    assert rel <= (1e-12 if fp64 else 5e-6)
    _, e1, g1, _ = _run(n, reps, ent, ham, th[1:2], fp64, mask=mask[1:2])
    assert e1[0] == e[1] and np.array_equal(g1[0], g[1])


@pytest.mark.parametrize("n,reps,ent,batch", [(14, 1, gv.GVQE_ENT_LINEAR, 2), (15, 3, gv.GVQE_ENT_CIRCULAR, 1),
                                              (16, 4, gv.GVQE_ENT_PAIRWISE, 3), (17, 5, gv.GVQE_ENT_FULL, 2),
                                              (19, 2, gv.GVQE_ENT_SCA, 2), (21, 5, gv.GVQE_ENT_LINEAR, 2)])
def test_xy_strings(n, reps, ent, batch):
    """X/Y strings as parts on the halves: 8 to 64 terms, even and odd numbers of Y on a
    half, parts shared by many strings, uneven halves; also no I/Z string at all."""
    for fraction in (0.6, 1.0):
        ham = wl.pauli_hamiltonian(n, 40 * n, seed=n, xy_fraction=fraction)
        th = wl.thetas(n, reps, batch, seed=n + 5)
        e0, e, g, _ = _run(n, reps, ent, ham, th, False)
        _, et, gt, _ = _run(n, reps, ent, ham, th, False, mps=-1)
        scale = ham.abs_sum()
        assert np.max(np.abs(e - et)) <= 1e-6 * scale and np.max(np.abs(e0 - et)) <= 1e-6 * scale
        rel = np.linalg.norm(g - gt) / np.linalg.norm(gt)
        print(f"n={n} reps={reps} ent={ent} xy={fraction}: vs tile passes grad {rel:.2e}, E {np.max(np.abs(e - et)) / scale:.1e}")
        assert rel <= 5e-6
        if n <= 16:
            with oracle.entangler(ent):
                er, gr = oracle.energy_grad(n, reps, th[0], ham.strings, ham.coeffs)
            assert abs(e[0] - er) <= 2e-5 * scale
            assert np.linalg.norm(g[0] - gr) <= 1e-4 * np.linalg.norm(gr)


@pytest.mark.parametrize("n,reps,ent", [(14, 1, gv.GVQE_ENT_LINEAR), (15, 3, gv.GVQE_ENT_REVERSE_LINEAR), (16, 2, gv.GVQE_ENT_CIRCULAR),
                                        (17, 4, gv.GVQE_ENT_PAIRWISE), (18, 2, gv.GVQE_ENT_SCA), (19, 5, gv.GVQE_ENT_FULL),
                                        (20, 3, gv.GVQE_ENT_LINEAR), (21, 3, gv.GVQE_ENT_LINEAR), (23, 2, gv.GVQE_ENT_LINEAR),
                                        (26, 3, gv.GVQE_ENT_LINEAR), (27, 2, gv.GVQE_ENT_LINEAR)])
def test_su2_layers(n, reps, ent):
    """Full EfficientSU2 layers (complex amplitudes, FP32): every register-round layout of the
    complex half circuits (8 to 15 index bits), uneven halves, 4 to 64 real terms, masks."""
    ham = wl.z_hamiltonian(n, 6 * n, seed=n)
    batch = 2
    P = 2 * n * (reps + 1)
    th = np.random.default_rng(n).uniform(-np.pi, np.pi, (batch, P))
    mask = wl.active_mask(P, batch, seed=n + 1)
    out = []
    for mps in (0, -1):
        a = gv.Ansatz(n, reps, entangler=ent, gates=gv.GVQE_GATES_RY_RZ)
        a.set_mps_layers(mps)
        h = gv.Hamiltonian.from_workload(ham)
        t = torch.as_tensor(th, device="cuda")
        e0 = gv.energy(a, h, t).cpu().numpy()
        e, g = gv.energy_grad(a, h, t, mask=torch.as_tensor(mask, device="cuda"))
        out.append((e0, e.cpu().numpy(), g.cpu().numpy()))
        assert ("terms" in a.describe()) == (mps == 0)
        a.close()
        h.close()
    (e0, e, g), (_, et, gt) = out
    scale = ham.abs_sum()
    assert np.all(g[mask == 0] == 0.0)
    assert np.max(np.abs(e - et)) <= 1e-6 * scale and np.max(np.abs(e0 - et)) <= 1e-6 * scale
    rel = np.linalg.norm(g - gt) / np.linalg.norm(gt)
    print(f"n={n} reps={reps} ent={ent}: vs tile passes grad {rel:.2e}, E {np.max(np.abs(e - et)) / scale:.1e}")
    assert rel <= 5e-6
    if n <= 16:
        with oracle.entangler(ent), oracle.gates(oracle.GATES_RY_RZ):
            er, gr = oracle.energy_grad(n, reps, th[0], ham.strings, ham.coeffs)
        gr = np.where(mask[0] == 1, gr, 0.0)
        assert abs(e[0] - er) <= 2e-5 * scale
        assert np.linalg.norm(g[0] - gr) <= 1e-4 * np.linalg.norm(gr)


@pytest.mark.parametrize("n,reps,ent,batch", [(10, 4, gv.GVQE_ENT_CIRCULAR, 1), (11, 4, gv.GVQE_ENT_SCA, 2), (12, 3, gv.GVQE_ENT_CIRCULAR, 1),
                                              (13, 4, gv.GVQE_ENT_CIRCULAR, 1), (16, 4, gv.GVQE_ENT_CIRCULAR, 1),
                                              (15, 3, gv.GVQE_ENT_SCA, 1), (12, 4, gv.GVQE_ENT_CIRCULAR, 64)])
def test_fp64_many_terms(n, reps, ent, batch):
    """FP64 with 64 and 256 terms on small registers (a CTA per row of the contraction); with
    many vectors the tile passes keep the call."""
    ham = wl.z_hamiltonian(n, 8 * n, seed=n)
    th = wl.thetas(n, reps, batch, seed=n)
    e0, e, g, _ = _run(n, reps, ent, ham, th, True)
    _, et, gt, _ = _run(n, reps, ent, ham, th, True, mps=-1)
    scale = ham.abs_sum()
    assert np.max(np.abs(e - et)) <= 1e-12 * scale and np.max(np.abs(e0 - et)) <= 1e-12 * scale
    assert np.linalg.norm(g - gt) <= 1e-12 * np.linalg.norm(gt)
    with oracle.entangler(ent):
        er, gr = oracle.energy_grad(n, reps, th[0], ham.strings, ham.coeffs)
    assert abs(e[0] - er) <= 1e-10 * scale and np.max(np.abs(g[0] - gr)) <= 1e-9 * scale


@pytest.mark.parametrize("n,reps,ent,batch,xy", [(18, 4, gv.GVQE_ENT_CIRCULAR, 35, 0), (19, 5, gv.GVQE_ENT_SCA, 16, 0),
                                                 (20, 4, gv.GVQE_ENT_SCA, 9, 0.4), (23, 4, gv.GVQE_ENT_CIRCULAR, 1, 0),
                                                 (24, 5, gv.GVQE_ENT_CIRCULAR, 1, 0), (25, 7, gv.GVQE_ENT_SCA, 2, 0)])
def test_energies_with_the_leading_layers_from_halves(n, reps, ent, batch, xy):
    # FP32 energies of circuits with more than 64 terms: the state after layer 3 (64 terms) comes from the halves.
    # Each amplitude is within a few 2^-23 of its value on either route: 2e-6 of sum |c| against FP64.
    ham = wl.pauli_hamiltonian(n, 6 * n, seed=n, xy_fraction=xy) if xy else wl.z_hamiltonian(n, 6 * n, seed=n)
    th = torch.as_tensor(wl.thetas(n, reps, batch, seed=n + ent), device="cuda")
    h = gv.Hamiltonian.from_workload(ham)
    a, b = gv.Ansatz(n, reps, entangler=ent), gv.Ansatz(n, reps, entangler=ent)
    b.set_mps_layers(-1)
    assert "state after layer 3" in a.describe() and "64 terms" in a.describe()
    assert "state after layer" not in b.describe()
    e, ep = gv.energy(a, h, th).cpu().numpy(), gv.energy(b, h, th).cpu().numpy()
    e64 = gv.energy(a, h, th, fp64=True).cpu().numpy()
    tol = 2e-6 * ham.abs_sum()
    assert np.abs(e - e64).max() <= tol and np.abs(ep - e64).max() <= tol
    assert np.array_equal(e, gv.energy(a, h, th).cpu().numpy())
    a.close()
    b.close()
    h.close()


@pytest.mark.parametrize("n,fp64,grad", [(14, True, True), (23, False, False)])
def test_falls_back_to_stored_states_under_a_memory_limit(n, fp64, grad):
    # 256 terms need more than the stored states they stand for: with room for those alone, the call runs on them
    reps, ent = 4, gv.GVQE_ENT_CIRCULAR
    h = gv.Hamiltonian.from_workload(wl.z_hamiltonian(n, 4 * n, seed=n))
    t = torch.as_tensor(wl.thetas(n, reps, 1, seed=n), device="cuda")

    def run(mps):
        a = gv.Ansatz(n, reps, entangler=ent)
        a.set_mps_layers(mps)
        out = gv.energy_grad(a, h, t, fp64=fp64) if grad else (gv.energy(a, h, t, fp64=fp64),)
        torch.cuda.synchronize()
        used = gv._lib.gvqe_device_memory_in_use()
        a.close()
        return [x.cpu() for x in out], used

    run(0)  # (its tables)
    passes, used = run(-1)
    free, more = run(0)
    assert more > used + (1 << 18)
    try:
        gv._lib.gvqe_set_device_memory_limit(used + (1 << 18))
        limited, _ = run(0)
    finally:
        gv._lib.gvqe_set_device_memory_limit(0)
    assert all(torch.equal(x, y) for x, y in zip(limited, passes))
    assert not all(torch.equal(x, y) for x, y in zip(free, passes))
    h.close()


def test_uneven_halves_of_the_largest_register():
    # 29 qubits: a half of 15 (two chunks a state) beside one of 14 in the same launches
    n, reps = 29, 3
    ham = wl.z_hamiltonian(n, 300, seed=n)
    th = wl.thetas(n, reps, 1, seed=n)
    e0, e, g, d = _run(n, reps, gv.GVQE_ENT_LINEAR, ham, th, False)
    assert "8 terms" in d
    _, et, gt, _ = _run(n, reps, gv.GVQE_ENT_LINEAR, ham, th, False, mps=-1)
    assert abs(e[0] - et[0]) <= 1e-7 * ham.abs_sum() and abs(e0[0] - et[0]) <= 1e-7 * ham.abs_sum()
    assert np.linalg.norm(g - gt) <= 5e-6 * np.linalg.norm(gt)


@pytest.mark.parametrize("n,reps,ent", [(16, 1, gv.GVQE_ENT_LINEAR), (18, 2, gv.GVQE_ENT_CIRCULAR), (20, 5, gv.GVQE_ENT_PAIRWISE),
                                        (19, 6, gv.GVQE_ENT_LINEAR)])
def test_fp32_gradients_are_not_short(n, reps, ent):
    # The tensor cores' accumulators round toward zero: 8 full-size steps a tile take 4.5 x 4.3e-8 of it, lambda's
    # cut 7.5e-8, S's steps 0.4 to 1.1e-7 (against 0.9 to 2.2e-7 of the norm), in all 1.6 to 2.7e-7 of every gradient unless
    # it is put back.  The other errors have no sign: 7e-8 a vector, 1e-8 in the mean of 64.
    ham = wl.z_hamiltonian(n, 40 * n, seed=n)
    th = wl.thetas(n, reps, 64, seed=n + 1).astype(np.float32).astype(np.float64)
    h = gv.Hamiltonian.from_workload(ham)
    a = gv.Ansatz(n, reps, entangler=ent)
    t = torch.as_tensor(th, device="cuda")
    g = gv.energy_grad(a, h, t)[1].cpu().numpy()
    g64 = gv.energy_grad(a, h, t, fp64=True)[1].cpu().numpy()
    short = np.mean(np.sum((g - g64) * g64, axis=1) / np.sum(g64 * g64, axis=1))
    print(f"n={n} reps={reps} ent={ent}: common factor off by {short:.1e}")
    assert abs(short) <= 1.2e-7
    a.close()
    h.close()
