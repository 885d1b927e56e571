"""The two-species FP32 step at tau = 1 on either side of the rule that says which lattices are held as
moments, and its streaming pass with columns of several layers, cut ragged, between moving walls and
periodic, against the 3-D oracle."""
import numpy as np
import pytest
import torch

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL32 = 1e-4  # the FP32 contract on rho and u


@pytest.fixture(scope="module")
def ref3d():
    from oracle import ref3d as R

    R.build()
    return R


def plan(nx, ny, nz):
    """(layers a block of the streaming pass walks, held as moments), as lbm3_create has them."""
    slots = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    columns = -(-nx // 32) * -(-ny // 4)
    chunk = min(range(1, 65), key=lambda k: (-(-columns * -(-nz // k) // slots) * (k + 2), k))
    return chunk, columns * nz <= slots or 2 * columns * nz > 3 * slots


def height(nx, ny, chunk, moments):
    """The smallest nz of that plan which chunk does not divide (chunk 1: any)."""
    return next(nz for nz in range(2, 400) if plan(nx, ny, nz) == (chunk, moments) and (chunk == 1 or nz % chunk))


@pytest.mark.parametrize("zbc", [0, 1])
@pytest.mark.parametrize("nx,ny,chunk,moments", [(64, 30, 1, True), (40, 34, 2, False), (64, 30, 2, True), (70, 45, 3, True),
                                                 (64, 61, 5, True), (96, 96, 7, True)])
def test_columns_match_oracle(ref3d, nx, ny, chunk, moments, zbc):
    nz = height(nx, ny, chunk, moments)
    prm = dict(W.EMULSION_PARAMS, body_force=1e-5, wall_u=(-0.01, 0.02))
    rho, _ = W.sphere_packing(nx, ny, nz, 0.4, seed=nz, r_mean=3, r_spread=1, periodic_z=not zbc)
    keys = ("tau", "G1", "G2", "G_AB", "rho0", "weight_norm", "body_force", "wall_u")
    ref = ref3d.RefLattice3D(nx, ny, nz, 2, **dict({k: prm[k] for k in keys if k in prm}, zbc=zbc))
    ref.set_fields(rho)
    lat = L.Lattice3(nx, ny, nz, 2, L.LBM_FP32, zbc, **prm)
    lat.set_fields(rho)
    records = torch.zeros((3, 5), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    lat.step(3)
    lat.step_totals(3, records)
    ref.step(6)
    r_rho, r_u, r_f = ref.fields()
    g_rho, g_u, g_f = lat.fields()
    assert np.abs(g_rho - r_rho).max() <= TOL32 * np.abs(r_rho).max()
    assert np.abs(g_f - r_f).max() <= TOL32 * np.abs(r_f).max()
    assert np.abs(g_u - r_u).max() <= TOL32 * np.abs(r_u).max() + 1e-7
    mass = records[2, :2].cpu().numpy()
    assert np.abs(mass - r_rho.sum(axis=(1, 2, 3))).max() <= TOL32 * mass.max()


@pytest.mark.parametrize("nx,ny,nz", [(48, 40, 40), (96, 64, 64)])
def test_mass_and_momentum_over_a_long_run(nx, ny, nz):
    """Mass and momentum of a periodic undriven emulsion over 4000 steps, held as populations (the first
    lattice) and as moments.  Every step rounds each
    site's sums to FP32; roundings without a direction add up as a random walk, so the mean
    density may move by a few 2^-24 at most.  A scale of 1 + 7e-9 a step (1/36 rounded to FP32) would
    move it by 2.8e-5, and the bound is a tenth of that."""
    rho, _ = W.sphere_packing(nx, ny, nz, 0.45, seed=5, r_mean=6, r_spread=2)
    lat = L.Lattice3(nx, ny, nz, 2, L.LBM_FP32, 0, **W.EMULSION_PARAMS)
    lat.set_fields(rho)
    m0, j0 = lat.totals()
    lat.step(4000)
    m1, j1 = lat.totals()
    sites = nx * ny * nz
    assert np.abs(m1 - m0).max() <= 2.8e-6 * sites
    assert np.abs(j1 - j0).max() <= 2.8e-6 * sites
