"""The FP64 step with tiles of 8 rows and of 4, each on lattices that its tiles do not divide in either
direction (sizes found from the device's SM count), against the oracle."""
import numpy as np
import pytest
import torch

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def tile_rows(nx, nz):
    """The rule of the PULL kernel for FP64 tiles (pull_tile_rows), for one lattice."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    most = [-(-(-(-nx // 32) * -(-nz // r)) // sm) * r for r in (8, 4)]
    return 4 if most[1] * 11 < most[0] * 10 else 8


def size(rows):
    return next((nx, nz) for nz in range(21, 140) for nx in range(105, 1500, 97)
                if nz % rows and nx % 32 and tile_rows(nx, nz) == rows and nx * nz > 12000)


@pytest.mark.parametrize("rows", [8, 4])
@pytest.mark.parametrize("ns,zbc", [(2, 1), (2, 0), (1, 1)])
def test_ragged_tiles_of_both_heights_match_oracle(oracle, rows, ns, zbc):
    nx, nz = size(rows)
    assert tile_rows(nx, nz) == rows and nz % rows and nx % 32
    prm = dict(W.EMULSION_PARAMS if ns == 2 else W.FILM_PARAMS, tau=(0.9, 1.1), body_force=1e-6, wall_u=(-0.01, 0.01))
    rho = W.noise_field(nx, nz, seed=rows, mean=0.8, amp=0.2, n_species=ns)
    ref = oracle.RefLattice(nx, nz, ns, zbc, **prm)
    ref.set_fields(rho)
    ref.step(12)
    lat = L.Lattice(nx, nz, ns, L.LBM_FP64, zbc, **prm)
    lat.set_fields(rho)
    lat.set_observe(1)
    lat.step(12)
    r_rho, r_u, r_f = ref.fields()[:3]
    g_rho, g_u, g_f = lat.fields()
    assert np.abs(g_rho - r_rho).max() <= 1e-12 * np.abs(r_rho).max()
    assert np.abs(g_f - r_f).max() <= 1e-12 * np.abs(r_f).max()
    assert np.abs(g_u - r_u).max() <= 1e-12 * np.abs(r_u).max() + 100 * EPS
    a, b = lat.observables(), ref.observables()
    for k in ("ux_z", "rho_z", "sxz_z", "ps_x", "pxx_x"):
        assert np.abs(a[k] - b[k]).max() <= 1e-12 * max(1.0, np.abs(b[k]).max()), k
