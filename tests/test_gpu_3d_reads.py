"""lbm3_get_fields tests the densities it reads, whatever form the state is held in: a state that the
last step broke is reported by the read that follows it, not only by the step after."""
import ctypes

import numpy as np
import pytest

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [L.LBM_FP32, L.LBM_FP64])
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("ns", [1, 2])
@pytest.mark.parametrize("shape", [(20, 9, 11), (96, 80, 72)])
def test_a_read_reports_the_density_the_last_step_broke(shape, ns, tau, precision):
    """A block of twice the attraction's contrast: the oracle's densities stay above 0.02 in the first
    step and fall below -2.8 in the second, at both relaxation times and numbers of species."""
    nx, ny, nz = shape
    rho = np.ones((ns, nz, ny, nx))
    rho[:, 4:6, 3:6, 8:12] = 1.5
    prm = dict(W.EMULSION_PARAMS if ns == 2 else W.SINGLE_PARAMS, G1=(-80.0, -80.0), G2=(0.0, 0.0), tau=(tau, tau))
    out = [np.empty((ns, nz, ny, nx)), np.empty((3, nz, ny, nx)), np.empty((ns, 19, nz, ny, nx))]
    for wanted in ((True, False, False), (False, True, False), (False, False, True), (True, True, True)):
        lat = L.Lattice3(nx, ny, nz, ns, precision, 0, **prm)
        lat.set_fields(rho)
        p = [ctypes.c_void_p(a.ctypes.data) if w else None for a, w in zip(out, wanted)]
        read = lambda: L.load().lbm3_get_fields(lat.h, *p, L.LBM_HOST)
        lat.step(1)
        assert read() == L.LBM_OK
        if wanted[0]:
            assert out[0].min() > 0.0
        lat.step(1)
        assert read() == L.LBM_ENONFINITE
        lat.set_fields(rho)  # a new state is clean
        assert read() == L.LBM_OK
