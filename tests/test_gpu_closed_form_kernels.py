"""The closed-form layers' kernels (gvqe_mps.cu) by their launches.  At the default options a diagonal H with
few layers is evaluated from the register's halves, so an explicit layer count, min(4, reps - 1), which is
what auto takes, runs them here; the event profiler's counts say that it did.  Tolerances as in test_gpu_mps.py."""
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

K_FWD, K_MPS, K_MPS_GRAD, K_CUT = 0, 5, 7, 11  # gvqe_engine.cuh, PassKind


def _run(n, reps, ham, th, ent, mps, tensor=0, mask=None):
    a = gv.Ansatz(n, reps, entangler=ent)
    a.set_mps_layers(mps)
    a.set_mps_tensor(tensor)
    h = gv.Hamiltonian.from_workload(ham)
    t = torch.as_tensor(th, device="cuda")
    m = None if mask is None else torch.as_tensor(mask, device="cuda")
    _lib.gvqe_profile_reset()
    _lib.gvqe_profile_enable(True)
    try:
        e0 = gv.energy(a, h, t).cpu().numpy()
        e, g = gv.energy_grad(a, h, t, mask=m)
        torch.cuda.synchronize()
    finally:
        _lib.gvqe_profile_enable(False)
    k = [_lib.gvqe_profile_read(x)["launches"] for x in (K_MPS, K_MPS_GRAD, K_FWD, K_CUT)]
    a.close()
    h.close()
    return e0, e.cpu().numpy(), g.cpu().numpy(), k


@pytest.mark.parametrize("n,reps,ent,batch,xy", [
    (14, 2, gv.GVQE_ENT_LINEAR, 7, 0), (15, 3, gv.GVQE_ENT_FULL, 2, 0), (17, 5, gv.GVQE_ENT_REVERSE_LINEAR, 2, 0),
    (19, 4, gv.GVQE_ENT_LINEAR, 2, 0), (16, 3, gv.GVQE_ENT_LINEAR, 2, 0.4), (22, 4, gv.GVQE_ENT_FULL, 2, 0)])
def test_leading_layers_in_closed_form(n, reps, ent, batch, xy):
    ham = wl.pauli_hamiltonian(n, 6 * n + 5, seed=n, xy_fraction=xy) if xy else wl.z_hamiltonian(n, 6 * n + 5, seed=n)
    th = wl.thetas(n, reps, batch, seed=n + reps)
    mask = wl.active_mask(n * (reps + 1), batch, seed=n + 1)
    mask[0, : 2 * n] = 0
    e0, e, g, k = _run(n, reps, ham, th, ent, min(4, reps - 1), mask=mask)
    assert k[0] > 0 and k[1] > 0 and k[2] > 0 and k[3] == 0
    e0t, et, gt, kt = _run(n, reps, ham, th, ent, -1, mask=mask)
    assert kt[0] == 0 and kt[1] == 0 and kt[2] > 0 and kt[3] == 0
    scale = ham.abs_sum()
    assert np.max(np.abs(e - et)) <= 2e-5 * scale and np.max(np.abs(e0 - e0t)) <= 2e-5 * scale
    assert np.all(g[mask == 0] == 0.0)
    assert np.linalg.norm(g - gt) <= 1e-4 * np.linalg.norm(gt)
    if n <= 17:
        with oracle.entangler(ent):
            er, gr = oracle.energy_grad(n, reps, th[0], ham.strings, ham.coeffs)
        gr = np.where(mask[0] == 1, gr, 0.0)
        assert abs(e[0] - er) <= 2e-5 * scale and np.linalg.norm(g[0] - gr) <= 1e-4 * np.linalg.norm(gr)


@pytest.mark.parametrize("n,reps,batch,ent", [(17, 5, 2, gv.GVQE_ENT_LINEAR), (21, 6, 3, gv.GVQE_ENT_FULL),
                                              (25, 5, 3, gv.GVQE_ENT_LINEAR), (26, 5, 2, gv.GVQE_ENT_LINEAR),
                                              (23, 5, 1, gv.GVQE_ENT_REVERSE_LINEAR)])
def test_bond_16_kernels_on_the_tensor_cores_and_the_fp32_pipe(n, reps, batch, ent):
    ham = wl.z_hamiltonian(n, 4 * n, seed=n)
    th = wl.thetas(n, reps, batch, seed=300 + n)
    e_tc, _, g_tc, k = _run(n, reps, ham, th, ent, 4, 0)
    assert k[0] > 0 and k[1] > 0 and k[3] == 0
    e_f, _, g_f, k = _run(n, reps, ham, th, ent, 4, -1)
    assert k[0] > 0 and k[1] > 0 and k[3] == 0
    e_t, _, g_t, _ = _run(n, reps, ham, th, ent, -1)
    assert not np.array_equal(g_tc, g_f)  # two kernels
    assert np.max(np.abs(e_tc - e_t)) <= 2e-5 * ham.abs_sum() and np.max(np.abs(e_f - e_t)) <= 2e-5 * ham.abs_sum()
    for b in range(batch):
        assert np.linalg.norm(g_tc[b] - g_f[b]) <= 1e-5 * np.linalg.norm(g_f[b])
        assert np.linalg.norm(g_tc[b] - g_t[b]) <= 1e-5 * np.linalg.norm(g_t[b])
