"""The 3-D FP32 step at tau = 1, whose state is held as moments: changes of the relaxation times and of
the wall velocities on the way (which expand it to populations), reads that leave the trajectory
alone, and the column lengths of its streaming pass, against the 3-D oracle."""
import numpy as np
import pytest

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL32 = 1e-4  # the FP32 contract on rho and u


@pytest.fixture(scope="module")
def ref3d():
    from oracle import ref3d as R

    R.build()
    return R


def rel(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


def ref_of(ref3d, shape, ns, zbc, prm):
    keys = ("tau", "G1", "G2", "G_AB", "rho0", "weight_norm", "body_force", "psi_form", "wall_u")
    return ref3d.RefLattice3D(*shape, ns, **dict({k: prm[k] for k in keys if k in prm}, zbc=zbc))


@pytest.mark.parametrize("ns", [1, 2])
@pytest.mark.parametrize("zbc,shape", [(1, (37, 13, 9)), (0, (33, 6, 70)), (1, (5, 3, 1))])
def test_changes_on_the_way_match_oracle(ref3d, ns, zbc, shape):
    nx, ny, nz = shape
    base = dict(W.EMULSION_PARAMS if ns == 2 else W.SINGLE_PARAMS, body_force=1e-5)
    phases = [dict(base, wall_u=(-0.01, 0.01)), dict(base, wall_u=(0.02, 0.0)), dict(base, wall_u=(0.02, 0.0), tau=(0.8, 0.9)),
              dict(base, wall_u=(0.02, 0.0)), dict(base, wall_u=(0.02, 0.0), G1=(-8.5, -7.5))]
    rho = 0.8 + 0.2 * (2.0 * W.uniform(nx + nz, ns * nx * ny * nz) - 1.0).reshape(ns, nz, ny, nx)
    lat = L.Lattice3(nx, ny, nz, ns, L.LBM_FP32, zbc, **phases[0])
    lat.set_fields(rho)
    f = None
    for prm in phases:
        ref = ref_of(ref3d, shape, ns, zbc, prm)
        ref.set_fields(rho) if f is None else ref.set_populations(f)
        lat.set_params(**prm)
        lat.step(4)
        ref.step(4)
        r_rho, r_u, f = ref.fields()
        g_rho, g_u, g_f = lat.fields()
        assert rel(g_rho, r_rho) <= TOL32 and rel(g_f, f) <= TOL32
        assert np.abs(g_u - r_u).max() <= TOL32 * np.abs(r_u).max() + 1e-7


def test_reads_and_totals_leave_the_trajectory_alone():
    nx, ny, nz = 41, 18, 23
    rho, _ = W.sphere_packing(nx, ny, nz, 0.4, seed=3, r_mean=3, r_spread=1)
    a, b = [L.Lattice3(nx, ny, nz, 2, L.LBM_FP32, 0, **W.EMULSION_PARAMS) for _ in range(2)]
    for lat in (a, b):
        lat.set_fields(rho)
    a.step(9)
    for n in (0, 1, 3, 5):
        b.step(n)
        b.fields()
        b.totals()
    assert all(np.array_equal(p, q) for p, q in zip(a.fields(), b.fields()))


def test_fields_into_device_memory_are_those_of_the_host():
    """All of them and one alone, written by the kernels themselves."""
    import ctypes
    import torch

    nx, ny, nz = 21, 10, 7
    for precision in (L.LBM_FP32, L.LBM_FP64):
        rho = 0.9 + 0.1 * W.uniform(5, 2 * nx * ny * nz).reshape(2, nz, ny, nx)
        lat = L.Lattice3(nx, ny, nz, 2, precision, 1, **W.EMULSION_PARAMS)
        lat.set_fields(rho)
        lat.step(3)
        host = lat.fields()
        dev = [torch.zeros(h.shape, dtype=torch.float64, device="cuda") for h in host]
        torch.cuda.synchronize()
        p = [ctypes.c_void_p(t.data_ptr()) for t in dev]
        assert L.load().lbm3_get_fields(lat.h, *p, L.LBM_DEVICE) == L.LBM_OK
        assert all(np.array_equal(t.cpu().numpy(), h) for t, h in zip(dev, host))
        only = torch.zeros(host[1].shape, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert L.load().lbm3_get_fields(lat.h, None, ctypes.c_void_p(only.data_ptr()), None, L.LBM_DEVICE) == L.LBM_OK
        assert np.array_equal(only.cpu().numpy(), host[1])
