"""FP64 step: both tile heights the pull kernel chooses between (4 rows where 8 leave SMs without
work), ragged edges of each, one and two species, walls and observables, against the FP64 oracle."""
import numpy as np
import pytest

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


# 600 x 64 and 610 x 61: 152 and 160 tiles of 32 x 8 on 152 SMs (8 rows at the first, 4 at the
# second); 33 x 5: a ragged tile in both directions
@pytest.mark.parametrize("ns,walls,nx,nz,form", [(2, 1, 600, 64, 0), (1, 0, 600, 64, 0), (2, 0, 610, 61, 0), (2, 1, 33, 5, 0),
                                                 (2, 1, 600, 64, 1)])
def test_fp64_step_and_observables(oracle, ns, walls, nx, nz, form):
    """FP64 contract 1e-12 (its derivation and the velocity's rounding floor as in
    test_gpu_parity.py), with the pseudopotential in fixed point (form 0) or plain (form 1)."""
    prm = dict(W.EMULSION_PARAMS if ns == 2 else W.FILM_PARAMS, tau=(0.9, 1.0), body_force=1e-6, wall_u=(-0.01, 0.01))
    if form == 1:
        prm.update(psi_form=1, rho0=(1.0, 1.0), G1=(-3.0, -3.0), G2=(2.0, 2.0))
    rho = 0.7 + 0.5 * (2.0 * W.uniform(nx + nz, ns * nx * nz) - 1.0).reshape(ns, nz, nx)
    ref = oracle.RefLattice(nx, nz, ns, walls, **prm)
    ref.set_fields(rho)
    lat = L.Lattice(nx, nz, ns, L.LBM_FP64, walls, **prm)
    lat.set_fields(rho)
    ref.step(12)
    lat.step(12)
    r_rho, r_u, r_f = ref.fields()
    g_rho, g_u, g_f = lat.fields()
    assert rel(g_rho, r_rho) <= 1e-12 and rel(g_f, r_f) <= 1e-12
    assert np.abs(g_u - r_u).max() <= 1e-12 * np.abs(r_u).max() + 1e-14
    a, b = lat.observables(), ref.observables()
    for k in ("rho_z", "pxx_x"):
        assert rel(a[k].reshape(b[k].shape), b[k]) <= 1e-12, k
    assert np.abs(a["sxz_z"] - b["sxz_z"]).max() <= 4e-12 * np.abs(b["pxx_x"]).max()
