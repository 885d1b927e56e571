"""The totals of a 3-D state at the edges of their passes' blocks and grids (rows that blocks of four
leave over, one column, more row segments than run at once), against sums of the exported
populations.

Bound: a site's sums over its 19 populations are formed in the context's precision, of the
deviations from the reference density in FP32, each of their at most 48 roundings (19 terms there, 19 in
the populations' own, the scalings) within 2^-24 (2^-53) of the site's sum of magnitudes."""
import numpy as np
import pytest

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu

C19 = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0], [-1, -1, 0],
                [1, -1, 0], [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1], [-1, 0, 1], [0, 1, 1], [0, -1, -1],
                [0, 1, -1], [0, -1, 1]], float)
W19 = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.mark.parametrize("precision", [L.LBM_FP32, L.LBM_FP64])
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("ns", [1, 2])
@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 5, 3), (70, 7, 21), (128, 3, 2), (31, 130, 47), (129, 66, 24)])
def test_totals_are_sums_of_the_populations(shape, ns, tau, precision):
    nx, ny, nz = shape
    rho = (0.8 + 0.3 * (2.0 * W.uniform(nx + ny + nz, ns * nx * ny * nz) - 1.0)).reshape(ns, nz, ny, nx)
    prm = dict(W.EMULSION_PARAMS if ns == 2 else W.SINGLE_PARAMS, body_force=1e-5, tau=(tau, tau))
    lat = L.Lattice3(nx, ny, nz, ns, precision, 0, **prm)
    lat.set_fields(rho)
    for _ in range(2):  # of the initial state, and after steps
        m, j = lat.totals()
        f = lat.fields()[2]
        ref = rho.mean(axis=(1, 2, 3)) if precision == L.LBM_FP32 else np.zeros(ns)
        size = np.abs(f - (W19[None, :] * ref[:, None])[:, :, None, None, None]).sum(axis=(1, 2, 3, 4))
        eps = 2.0 ** (-24 if precision == L.LBM_FP32 else -53)
        # the exported numbers and numpy's own sums: FP64 roundings of the whole sum
        own = 1e-13 * np.abs(f).sum()
        assert np.all(np.abs(m - f.sum(axis=(1, 2, 3, 4))) <= 48 * eps * size + own)
        assert np.all(np.abs(j - np.einsum("slzyx,lk->k", f, C19)) <= 48 * eps * size.sum() + own)
        lat.step(5)
