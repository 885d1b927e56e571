"""lbm_adjoint_sweep: the same bits with one buffer of states and with two, in order with the stream's
other work; and the adjoint step on lattices narrower than its stencil and at the edges of its tiles."""
import numpy as np
import pytest
import torch

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [L.LBM_FP32, L.LBM_FP64])
@pytest.mark.parametrize("nsteps", [[4], [3, 3], [5, 5, 5, 2]])
def test_two_buffers_give_the_bits_of_one(precision, nsteps):
    nx, nz = 45, 31
    dt = torch.float32 if precision == L.LBM_FP32 else torch.float64
    prm = dict(W.EMULSION_PARAMS, body_force=1e-5)
    rho = W.noise_field(nx, nz, seed=8, mean=0.7, amp=0.2, n_species=2)
    lam0 = torch.from_numpy(np.random.default_rng(2).standard_normal((2, 9, nz, nx))).to("cuda", dt)
    got = []
    for two in (False, True):
        lat = L.Lattice(nx, nz, 2, precision, L.LBM_PERIODIC, **prm)
        lat.set_fields(rho)
        snaps = []
        for n in nsteps:
            s = torch.empty(L.lbm_snapshot_bytes(lat.h), dtype=torch.uint8, device="cuda")
            L.lbm_snapshot(lat.h, s)
            snaps.append(s)
            lat.step(n)
        seg = [torch.empty((max(nsteps), 2, 9, nz, nx), dtype=dt, device="cuda") for _ in range(2)]
        lam, grad = lam0.clone(), torch.zeros(8, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        L.lbm_adjoint_sweep(lat.h, snaps, nsteps, seg[0], seg[1] if two else None, lam, grad)
        g_rho = torch.empty((2, nz, nx), dtype=torch.float64, device="cuda")
        L.lbm_adjoint_initial(lat.h, lam, g_rho)  # follows the sweep on the context's stream
        lat.synchronize()
        got.append([t.cpu().numpy() for t in (lam, grad, g_rho)])
    assert all(np.array_equal(a, b) for a, b in zip(*got))
    assert np.abs(got[0][2]).max() > 0


def test_sweep_refuses_bad_arguments():
    lat = L.Lattice(16, 16, 1, L.LBM_FP64, L.LBM_PERIODIC, **W.SINGLE_PARAMS)
    lat.set_fields(W.noise_field(16, 16, seed=1))
    lam, grad = torch.zeros((1, 9, 16, 16), dtype=torch.float64, device="cuda"), torch.zeros(8, dtype=torch.float64, device="cuda")
    seg = torch.zeros((2, 1, 9, 16, 16), dtype=torch.float64, device="cuda")
    snap = torch.zeros(L.lbm_snapshot_bytes(lat.h), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    with pytest.raises(L.LbmError):
        L.lbm_adjoint_sweep(lat.h, [snap], [-1], seg, None, lam, grad)
    with pytest.raises(L.LbmError):  # no snapshot of this context there
        L.lbm_adjoint_sweep(lat.h, [snap], [2], seg, seg.clone(), lam, grad)
    L.lbm_adjoint_sweep(lat.h, [], [], seg, None, lam, grad)


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("nx,nz,ns", [(1, 1, 2), (2, 3, 2), (3, 1, 1), (33, 5, 2), (32, 4, 2), (65, 2, 1)])
def test_adjoint_step_on_small_lattices_matches_oracle(oracle, nx, nz, ns, fp32):
    """Bounds as in test_gpu_adjoint.py's step: FP64 1e-12 of max |lam|, parameters 1e-10; FP32 5e-5 and
    1e-4, with the floor of the summed rounding."""
    prm = dict(W.EMULSION_PARAMS if ns == 2 else W.SINGLE_PARAMS, tau=(0.8, 1.2), body_force=1e-5)
    rho = W.noise_field(nx, nz, seed=nx + nz, mean=0.7, amp=0.3, n_species=ns)
    u = 0.02 * W.noise_field(nx, nz, seed=nx, mean=0.0, amp=1.0, n_species=2)
    ref = oracle.RefLattice(nx, nz, ns, 0, **prm)
    ref.set_fields(rho, u)
    ref.step(3)
    f = ref.fields()[2]
    lam_next = np.random.default_rng(nx).standard_normal(f.shape)
    lam_ref, grad_ref = ref.adjoint_step(lam_next)
    dt = np.float32 if fp32 else np.float64
    lat = L.Lattice(nx, nz, ns, L.LBM_FP64, L.LBM_PERIODIC, **prm)
    d = [torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).cuda() for a in (f, lam_next)]
    lam, grad = torch.empty_like(d[0]), torch.zeros(8, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    L.lbm_adjoint_step(lat.h, d[0], d[1], lam, grad)
    lat.synchronize()
    tol, rtol, atol = (5e-5, 1e-4, 1e-6) if fp32 else (1e-12, 1e-10, 1e-12)
    assert np.abs(lam.cpu().numpy() - lam_ref).max() <= tol * np.abs(lam_ref).max()
    atol *= nx * nz * np.abs(lam_next).max()
    g = grad.cpu().numpy()
    for k in range(8):
        assert abs(g[k] - grad_ref[k]) <= rtol * abs(grad_ref[k]) + atol, k
