"""Which evaluation a call takes, and that it has one to take: from the register's halves or
on stored states, told apart by the launches that the event profiler counts.  Results of the two are
compared in test_gpu_cut.py; where a call is moved from one to the other, its bits are the other's."""
import numpy as np
import pytest

from paper_2607_02749_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2607_02749_gb300 as gv  # noqa: E402
from paper_2607_02749_gb300 import _lib  # noqa: E402

K_FWD, K_BWD, K_CUT = 0, 1, 11  # gvqe_engine.cuh, PassKind


def _profiled(f, kinds):
    """f() and how many launches of each kind it made."""
    _lib.gvqe_profile_reset()
    _lib.gvqe_profile_enable(True)
    try:
        r = f()
        torch.cuda.synchronize()
    finally:
        _lib.gvqe_profile_enable(False)
    return r, [_lib.gvqe_profile_read(k)["launches"] for k in kinds]


def test_xy_strings_run_on_stored_states_where_their_parts_do_not_fit():
    # 10,000 parts of 64 terms take 3 GB, a state of 24 qubits 64 MiB: with 1.25 GiB left on the device (and no
    # declared limit) the call runs on stored states (pairwise: no closed-form layers, the same passes as -1)
    n, reps = 24, 6
    h = gv.Hamiltonian.from_workload(wl.pauli_hamiltonian(n, 20000, seed=3, xy_fraction=1.0, max_weight=8))
    t = torch.as_tensor(wl.thetas(n, reps, 1, seed=n), device="cuda")

    def run(mps):
        a = gv.Ansatz(n, reps, entangler=gv.GVQE_ENT_PAIRWISE)
        a.set_mps_layers(mps)
        e, k = _profiled(lambda: gv.energy(a, h, t), (K_CUT, K_FWD))
        a.close()
        return e.item(), k

    stored, k = run(-1)
    assert k[0] == 0 and k[1] > 0
    halves, k = run(0)
    assert k == [1, 0]
    torch.cuda.empty_cache()
    block = torch.empty(torch.cuda.mem_get_info()[0] - (5 << 28), dtype=torch.uint8, device="cuda")
    try:
        short, k = run(0)
    finally:
        del block
        torch.cuda.empty_cache()
    assert k[0] == 0 and k[1] > 0
    assert short == stored and halves != stored
    h.close()


@pytest.mark.parametrize("n,reps,ent,count,fp64", [(14, 3, gv.GVQE_ENT_CIRCULAR, 4, False), (10, 4, gv.GVQE_ENT_CIRCULAR, 1, True)])
def test_staged_batch_runs_on_stored_states_where_the_halves_do_not_fit(n, reps, ent, count, fp64):
    # 64 or 256 terms of a small register need more than its stored states: with room for those alone the batch runs on them
    hams = [gv.Hamiltonian.from_workload(wl.z_hamiltonian(n, 4 * n, seed=k)) for k in range(count)]
    params = [torch.as_tensor(wl.thetas(n, reps, 1, seed=k)[0], device="cuda") for k in range(count)]

    def run(mps):
        ans = [gv.Ansatz(n, reps, entangler=ent) for _ in range(count)]
        for a in ans:
            a.set_mps_layers(mps)
        b = gv.Batch(ans, hams, fp64=fp64)
        grads = [torch.empty_like(p) for p in params]
        e = b.run(params, grads=grads)
        torch.cuda.synchronize()
        used = _lib.gvqe_device_memory_in_use()
        for x in [b] + ans:
            x.close()
        return [e.cpu()] + [g.cpu() for g in grads], used

    run(-1)  # (the Hamiltonians' tables)
    stored, used = run(-1)
    halves, more = run(0)
    assert more > used + (1 << 18)
    try:
        _lib.gvqe_set_device_memory_limit(used + (1 << 18))
        limited, _ = run(0)
    finally:
        _lib.gvqe_set_device_memory_limit(0)
    assert all(torch.equal(x, y) for x, y in zip(limited, stored))
    assert not all(torch.equal(x, y) for x, y in zip(halves, stored))
    for h in hams:
        h.close()


@pytest.mark.parametrize("xy", [0.0, 0.4])
def test_autotuner_times_the_passes_it_chooses_between(xy):
    # the evaluation itself takes the halves, which read no tile plan: every candidate must run its passes
    n, reps = 17, 2
    h = gv.Hamiltonian.from_workload(wl.pauli_hamiltonian(n, 30, seed=1, xy_fraction=xy))
    t = torch.as_tensor(wl.thetas(n, reps, 1, seed=2), device="cuda")
    a = gv.Ansatz(n, reps, entangler=gv.GVQE_ENT_PAIRWISE)
    rep, k = _profiled(lambda: a.autotune(h, t, cache=None), (K_CUT, K_FWD, K_BWD))
    candidates = rep.count(" ms") - 1
    assert candidates >= 2
    assert k[0] == 0 and k[1] >= 2 * candidates and k[2] >= 2 * candidates, (rep, k)
    if not xy:
        assert _profiled(lambda: gv.energy_grad(a, h, t), (K_CUT, K_FWD))[1] == [1, 0]
    a.close()
    h.close()


@pytest.mark.parametrize("option", ["tile_bits", "split", "xy_tile_bits"])
@pytest.mark.parametrize("fp64", [False, True])
def test_tile_options_name_the_passes_that_run(option, fp64):
    # an option that says how stored states are cut is honoured by the call it is set for
    n, reps = 18, 2
    xy = option == "xy_tile_bits"
    h = gv.Hamiltonian.from_workload(wl.pauli_hamiltonian(n, 700, seed=n, xy_fraction=0.4 if xy else 0.0))
    t = torch.as_tensor(wl.thetas(n, reps, 1, seed=5), device="cuda")
    a = gv.Ansatz(n, reps, **({} if xy else {"tile_bits": 11} if option == "tile_bits" else {"split": 2}))
    if xy:
        _lib.gvqe_ansatz_set_option(a.handle, _lib.GVQE_OPT_XY_TILE_BITS, 11)
    _, k = _profiled(lambda: gv.energy_grad(a, h, t, fp64=fp64), (K_CUT, K_FWD, K_BWD))
    assert k[0] == 0 and k[1] > 0 and k[2] > 0
    _lib.gvqe_ansatz_set_option(a.handle, {"tile_bits": 1, "split": 3}.get(option, _lib.GVQE_OPT_XY_TILE_BITS), 0)
    if not (fp64 and xy):
        assert _profiled(lambda: gv.energy(a, h, t, fp64=fp64), (K_CUT, K_FWD))[1] == [1, 0]
    a.close()
    h.close()


@pytest.mark.parametrize("n,reps,ent,batch,grad,cut", [
    (12, 6, gv.GVQE_ENT_LINEAR, 128, True, 0),    # 64 terms: 1274 us from the halves, 654 on stored states
    (12, 6, gv.GVQE_ENT_LINEAR, 1, True, 1),      # 107, 645
    (10, 2, gv.GVQE_ENT_CIRCULAR, 1024, False, 0),  # 16 terms: 250, 158
    (10, 2, gv.GVQE_ENT_CIRCULAR, 16, False, 1),  # 52, 119
    (14, 6, gv.GVQE_ENT_LINEAR, 256, True, 1),    # 64 terms: 4178, 4417
    (16, 5, gv.GVQE_ENT_LINEAR, 64, False, 1),    # 32 terms: 483, 1380
    (12, 2, gv.GVQE_ENT_LINEAR, 1024, True, 1),   # 4 terms: 404, 1260
    (17, 4, gv.GVQE_ENT_CIRCULAR, 1, True, 0)])   # 256 terms: 1326, 650
def test_fp64_calls_take_the_faster_evaluation(n, reps, ent, batch, grad, cut):
    _faster(n, reps, ent, batch, grad, cut, True, 1e-12, 1e-12)


# us from the halves and on stored states at 512 vectors: 465 and 149, 889 and 362; 591 and 221; 863 and 700; else the halves
@pytest.mark.parametrize("n,reps,ent,batch,grad,cut", [
    (14, 3, gv.GVQE_ENT_CIRCULAR, 512, False, 0), (14, 3, gv.GVQE_ENT_CIRCULAR, 512, True, 0),
    (14, 3, gv.GVQE_ENT_CIRCULAR, 8, True, 1), (15, 3, gv.GVQE_ENT_SCA, 512, False, 0),
    (16, 6, gv.GVQE_ENT_PAIRWISE, 512, False, 0), (16, 6, gv.GVQE_ENT_PAIRWISE, 1, False, 1),
    (14, 6, gv.GVQE_ENT_LINEAR, 512, True, 1), (18, 3, gv.GVQE_ENT_CIRCULAR, 64, True, 1),
    (14, 1, gv.GVQE_ENT_LINEAR, 512, True, 1)])
def test_fp32_calls_take_the_faster_evaluation(n, reps, ent, batch, grad, cut):
    _faster(n, reps, ent, batch, grad, cut, False, 1e-6, 5e-6)


@pytest.mark.parametrize("n,reps,ent,batch,strings,grad,cut", [
    (14, 3, gv.GVQE_ENT_CIRCULAR, 1, 2800, True, 0),  # 1148 us from the halves, 288 on stored states
    (16, 2, gv.GVQE_ENT_LINEAR, 1, 80, True, 0),      # 160, 143
    (18, 6, gv.GVQE_ENT_LINEAR, 8, 3600, False, 0),   # 1334, 463
    (20, 2, gv.GVQE_ENT_LINEAR, 8, 4000, True, 1),    # 506, 1259
    (24, 2, gv.GVQE_ENT_CIRCULAR, 1, 960, True, 1),   # 483, 1264
    (16, 4, gv.GVQE_ENT_LINEAR, 1, 640, False, 1),    # 113, 149
    # the halves' kernels at every number of terms they are built for (8 to 64)
    (14, 6, gv.GVQE_ENT_LINEAR, 16, 28, True, 1), (15, 6, gv.GVQE_ENT_FULL, 16, 30, True, 1),
    (21, 5, gv.GVQE_ENT_LINEAR, 8, 840, True, 1), (22, 1, gv.GVQE_ENT_LINEAR, 4, 880, True, 1),
    (22, 2, gv.GVQE_ENT_CIRCULAR, 4, 880, True, 1), (23, 3, gv.GVQE_ENT_REVERSE_LINEAR, 4, 920, True, 1),
    (24, 6, gv.GVQE_ENT_REVERSE_LINEAR, 1, 500, True, 1), (25, 2, gv.GVQE_ENT_PAIRWISE, 2, 2000, True, 1)])
def test_xy_calls_take_the_faster_evaluation(n, reps, ent, batch, strings, grad, cut):
    _faster(n, reps, ent, batch, grad, cut, False, 1e-6, 5e-6, strings)


def _faster(n, reps, ent, batch, grad, cut, fp64, tol_e, tol_g, xy=0):
    # by the terms and the vectors of the call; both within rounding of each other at either choice (tolerances of test_gpu_cut.py)
    ham = wl.pauli_hamiltonian(n, xy, seed=n) if xy else wl.z_hamiltonian(n, 5 * n, seed=n)
    h = gv.Hamiltonian.from_workload(ham)
    t = torch.as_tensor(wl.thetas(n, reps, batch, seed=n + reps), device="cuda")
    out = []
    for mps in (0, -1):
        a = gv.Ansatz(n, reps, entangler=ent)
        a.set_mps_layers(mps)
        f = (lambda: gv.energy_grad(a, h, t, fp64=fp64)) if grad else (lambda: (gv.energy(a, h, t, fp64=fp64),))
        r, k = _profiled(f, (K_CUT, K_FWD))
        assert (k[0] > 0) == (cut == 1 and mps == 0) and (k[1] > 0) == (k[0] == 0), k
        out.append([x.cpu().numpy() for x in r])
        a.close()
    assert np.abs(out[0][0] - out[1][0]).max() <= tol_e * ham.abs_sum()
    if grad:
        assert np.linalg.norm(out[0][1] - out[1][1]) <= tol_g * np.linalg.norm(out[1][1])
    h.close()


@pytest.mark.parametrize("n,reps,ent,batch", [(14, 4, gv.GVQE_ENT_CIRCULAR, 512), (17, 7, gv.GVQE_ENT_PAIRWISE, 64)])
def test_leading_layers_of_small_registers_run_as_passes(n, reps, ent, batch):
    # 529 us with them from the halves, 184 with passes; 307 and 279: one route and its bits, at every option
    h = gv.Hamiltonian.from_workload(wl.z_hamiltonian(n, 5 * n, seed=n))
    t = torch.as_tensor(wl.thetas(n, reps, batch, seed=n), device="cuda")
    out = []
    for mps in (0, -1):
        a = gv.Ansatz(n, reps, entangler=ent)
        a.set_mps_layers(mps)
        out.append(gv.energy(a, h, t))
        assert "state after layer" not in a.describe()
        a.close()
    assert torch.equal(*out)
    h.close()
