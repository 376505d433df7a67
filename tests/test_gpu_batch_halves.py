"""Staged batches at the default options: the register's halves over many different problems in
one launch (gvqe_cut.cuh, item lists).  Sizes: halves of 7 to 13 qubits, even and uneven, so that a group holds
both the small and the layer-by-layer half circuits, with circuits of fewer layers and fewer path bits that
leave a launch early; 16, 32 and 64 terms; every entangler; a Hamiltonian in several slots."""
import numpy as np
import pytest

import oracle
from paper_2607_02749_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2607_02749_gb300 as gv  # noqa: E402
from paper_2607_02749_gb300 import _lib  # noqa: E402

LI, CI, FU, RV, PW, SC = range(6)
# (n, reps, entangler): the groups are 16 terms (1 to 16), 32 and 64, by the larger half
SHAPES = {
    "small halves": [(14, 1, LI), (15, 4, FU), (17, 2, CI), (19, 3, RV), (20, 4, PW), (18, 5, LI), (16, 5, PW), (20, 6, FU), (18, 3, SC),
                     (19, 6, LI), (20, 3, CI)],
    "halves of 11 to 13": [(21, 1, LI), (21, 4, PW), (22, 2, SC), (22, 3, LI), (23, 4, FU), (24, 2, CI), (24, 1, RV), (25, 3, LI),
                           (21, 5, LI), (22, 5, RV), (24, 5, PW), (21, 3, CI), (22, 6, LI), (23, 3, SC), (24, 6, RV)],
}


@pytest.mark.parametrize("shapes", list(SHAPES))
@pytest.mark.parametrize("grad", [True, False])
def test_staged_batch_equals_single_calls(shapes, grad):
    insts = SHAPES[shapes] + SHAPES[shapes][:2]  # two problems again, on the first ones' Hamiltonians
    rng = np.random.default_rng(len(insts))
    hams = [wl.z_hamiltonian(n, 4 * n, seed=10 * n + r) for n, r, _ in insts[:-2]]
    hams += hams[:2]
    handles = [gv.Hamiltonian.from_workload(h) for h in hams[:-2]]
    handles += handles[:2]
    ans = [gv.Ansatz(n, r, entangler=e) for n, r, e in insts]
    thetas = [rng.uniform(-np.pi, np.pi, n * (r + 1)) for n, r, _ in insts]
    masks = [(rng.random(t.size) < 0.6).astype(np.uint8) for t in thetas]
    p = [torch.as_tensor(t, device="cuda") for t in thetas]
    m = [torch.as_tensor(x, device="cuda") for x in masks]
    b = gv.Batch(ans, handles)
    grads = [torch.full_like(x, float("nan")) for x in p] if grad else None
    for _ in range(2):  # the graph is replayed
        e = b.run(p, masks=m if grad else None, grads=grads).cpu().numpy()
    for k, (n, r, ent) in enumerate(insts):
        if grad:
            e1, g1 = gv.energy_grad(ans[k], handles[k], p[k], mask=m[k])
            assert torch.equal(grads[k], g1[0]), (n, r, ent)
        else:
            e1 = gv.energy(ans[k], handles[k], p[k])
        assert e[k] == e1.item(), (n, r, ent)
        # against stored states: the tolerances of test_gpu_cut.py
        a = gv.Ansatz(n, r, entangler=ent)
        a.set_mps_layers(-1)
        es, gs = gv.energy_grad(a, handles[k], p[k], mask=m[k])
        assert abs(e[k] - es.item()) <= 1e-7 * hams[k].abs_sum(), (n, r, ent)
        if grad:
            d = (grads[k] - gs[0]).norm().item() / max(gs[0].norm().item(), 1e-300)
            assert d <= 5e-6, (n, r, ent, d)
            assert np.all(grads[k].cpu().numpy()[masks[k] == 0] == 0.0)
            if n <= 15:
                with oracle.entangler(ent):
                    er, gr = oracle.energy_grad(n, r, thetas[k], hams[k].strings, hams[k].coeffs)
                assert abs(e[k] - er) <= 2e-5 * hams[k].abs_sum()
                assert np.linalg.norm(grads[k].cpu().numpy() - gr * masks[k]) <= 1e-4 * np.linalg.norm(gr)
        a.close()
    for x in [b] + ans + handles[:-2]:
        x.close()


@pytest.mark.parametrize("n,reps,ent,count,fp64,halves", [(15, 6, LI, 64, False, False), (14, 3, CI, 64, False, False), (16, 1, LI, 64, False, True),
                                                          (18, 3, CI, 16, False, True), (10, 2, CI, 256, True, False), (12, 2, LI, 64, True, True)])
def test_staged_batch_takes_the_faster_evaluation(n, reps, ent, count, fp64, halves):
    # as gvqe_energy does (test_gpu_halves_routes.py), by the work alone; on stored states the bits of that option
    handles = [gv.Hamiltonian.from_workload(wl.z_hamiltonian(n, 3 * n, seed=k)) for k in range(count)]
    p = [torch.as_tensor(t, device="cuda") for t in wl.thetas(n, reps, count, seed=n)]
    out = []
    for mps in (0, -1):
        ans = [gv.Ansatz(n, reps, entangler=ent) for _ in range(count)]
        for a in ans:
            a.set_mps_layers(mps)
        b = gv.Batch(ans, handles, fp64=fp64)
        out.append(b.run(p).cpu().numpy())
        for x in [b] + ans:
            x.close()
    assert np.array_equal(*out) == (not halves)
    for x in handles:
        x.close()


def test_staged_gradients_of_deep_circuits_stay_in_the_graph():
    # energies of these begin with a state written from the halves and run as single calls; gradients have no
    # such state (3193 us as four single calls, 2865 in the graph): one launch, the bits of a single call either way
    insts = [(23, 4, CI), (14, 2, LI), (23, 5, SC)]
    handles = [gv.Hamiltonian.from_workload(wl.z_hamiltonian(n, 3 * n, seed=n + r)) for n, r, _ in insts]
    ans = [gv.Ansatz(n, r, entangler=e) for n, r, e in insts]
    p = [torch.as_tensor(wl.thetas(n, r, 1, seed=n)[0], device="cuda") for n, r, _ in insts]
    grads = [torch.empty_like(x) for x in p]
    b = gv.Batch(ans, handles)
    b.run(p, grads=grads)
    before = _lib.gvqe_launch_count()
    e = b.run(p, grads=grads).cpu()
    assert _lib.gvqe_launch_count() - before == 1
    e0 = b.run(p).cpu()
    for k in range(len(insts)):
        e1, g1 = gv.energy_grad(ans[k], handles[k], p[k])
        assert e[k].item() == e1.item() and torch.equal(grads[k], g1[0])
        assert e0[k].item() == gv.energy(ans[k], handles[k], p[k]).item()
    for x in [b] + ans + handles:
        x.close()
