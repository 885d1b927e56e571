"""FP64 steps with couplings and weights far beyond any setting, which lbm_set_params accepts: the fixed-point
sums have no range for them, and the results are the FP64 forms', against the oracles."""
import numpy as np
import pytest
import torch

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu
KEYS = ("tau", "G1", "G2", "G_AB", "rho0", "weight_norm", "body_force")
TINY = (1e-300, 1e-310, 5e-324)


def rel(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


@pytest.mark.parametrize("tiny", TINY)
@pytest.mark.parametrize("ns", [1, 2])
def test_vanishing_couplings_2d(oracle, ns, tiny):
    nx, nz = 37, 21
    rho = W.noise_field(nx, nz, seed=3, mean=0.8, amp=0.3, n_species=ns)
    prm = dict(W.EMULSION_PARAMS if ns == 2 else W.SINGLE_PARAMS, G1=(-9 * tiny,) * 2, G2=(8 * tiny,) * 2, body_force=1e-5)
    ref = oracle.RefLattice(nx, nz, ns, 0, **prm)
    ref.set_fields(rho)
    ref.step(5)
    lat = L.Lattice(nx, nz, ns, L.LBM_FP64, L.LBM_PERIODIC, **prm)
    lat.set_fields(rho)
    lat.set_observe(1)
    lat.step(5)
    r_rho, r_u, r_f = ref.fields()[:3]
    g_rho, g_u, g_f = lat.fields()
    assert rel(g_rho, r_rho) <= 1e-12 and rel(g_f, r_f) <= 1e-12 and rel(g_u, r_u) <= 1e-12
    a, b = lat.observables(), ref.observables()
    for k in ("sxz_z", "ps_x", "pxx_x"):
        assert np.abs(a[k] - b[k]).max() <= 1e-12 * max(1.0, np.abs(b[k]).max()), k


@pytest.mark.parametrize("tiny", TINY)
def test_vanishing_couplings_3d(tiny):
    from oracle import ref3d as R

    R.build()
    nx, ny, nz = 18, 7, 9
    rho = (0.8 + 0.3 * (2 * W.uniform(5, 2 * nx * ny * nz) - 1)).reshape(2, nz, ny, nx)
    prm = dict(W.EMULSION_PARAMS, G1=(-9 * tiny,) * 2, G2=(8 * tiny,) * 2, body_force=1e-5)
    ref = R.RefLattice3D(nx, ny, nz, 2, **dict({k: prm[k] for k in KEYS if k in prm}, zbc=0))
    ref.set_fields(rho)
    ref.step(5)
    lat = L.Lattice3(nx, ny, nz, 2, L.LBM_FP64, 0, **prm)
    lat.set_fields(rho)
    lat.step(5)
    for g, r in zip(lat.fields(), ref.fields()):
        assert rel(g, r) <= 1e-12


@pytest.mark.parametrize("huge", [1e280, 1e300, 1.7e308])
def test_couplings_that_overflow_are_reported(huge):
    rho = W.noise_field(33, 18, seed=3, mean=0.8, amp=0.3, n_species=2)
    lat = L.Lattice(33, 18, 2, L.LBM_FP64, L.LBM_PERIODIC, **dict(W.EMULSION_PARAMS, G1=(-huge,) * 2, G2=(0.0, 0.0)))
    lat.set_fields(rho)
    lat.step(3)
    with pytest.raises(L.LbmError) as e:
        lat.synchronize()
    assert e.value.code == L.LBM_ENONFINITE
    lat3 = L.Lattice3(9, 6, 11, 2, L.LBM_FP64, 0, **dict(W.EMULSION_PARAMS, G1=(-huge,) * 2, G2=(0.0, 0.0)))
    lat3.set_fields(rho)
    lat3.step(3)
    with pytest.raises(L.LbmError) as e:
        lat3.synchronize()
    assert e.value.code == L.LBM_ENONFINITE


def test_adjoint_with_tiny_weights_and_large_couplings():
    """weight_norm scaled down and the couplings up by 2^950: the same forces, and every derivative the
    same but those of the couplings, smaller by that factor (powers of two: the FP64 forms keep the bits
    of their products, the other side's are in fixed point)."""
    nx, nz, by = 45, 20, 2.0 ** 950
    rho = W.noise_field(nx, nz, seed=8, mean=0.7, amp=0.3, n_species=2)
    lam_next = torch.from_numpy(np.random.default_rng(1).standard_normal((2, 9, nz, nx))).cuda()
    out = []
    for s in (1.0, by):
        p = dict(W.EMULSION_PARAMS, tau=(0.8, 1.2), body_force=1e-5)
        p = dict(p, G1=tuple(s * g for g in p["G1"]), G2=tuple(s * g for g in p["G2"]), G_AB=s * p["G_AB"],
                 weight_norm=p["weight_norm"] / s)
        lat = L.Lattice(nx, nz, 2, L.LBM_FP64, L.LBM_PERIODIC, **p)
        lat.set_fields(rho)
        f = torch.empty_like(lam_next)
        L.lbm_export_state(lat.h, f)
        lam, grad = torch.empty_like(f), torch.zeros(8, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        L.lbm_adjoint_step(lat.h, f, lam_next, lam, grad)
        lat.synchronize()
        g = grad.cpu().numpy()
        g[:5] *= s
        out.append((lam.cpu().numpy(), g))
    (la, ga), (lb, gb) = out
    assert np.abs(la - lb).max() <= 1e-12 * np.abs(la).max()
    assert np.all(np.abs(ga - gb) <= 1e-10 * np.abs(ga) + 1e-12 * nx * nz * 5)
