"""lbm_export_state from FP32 gives the stored values widened by the base weights and rounded once, and
passes infinite and NaN populations on as they are."""
import numpy as np
import pytest
import torch

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [L.LBM_KERNEL_PULL, L.LBM_KERNEL_FUSED])
def test_fp32_export_of_special_values(kernel):
    nx, nz = 37, 70
    lat = L.Lattice(nx, nz, 2, L.LBM_FP32, L.LBM_PERIODIC, kernel=kernel, **W.EMULSION_PARAMS)
    lat.set_fields(W.noise_field(nx, nz, seed=2, mean=0.8, amp=0.2, n_species=2))
    f = np.random.default_rng(4).uniform(1e-3, 0.5, (2, 9, nz, nx))
    special = {(0, 0, 3, 4): np.inf, (0, 5, 69, 36): -np.inf, (1, 2, 0, 0): np.nan, (1, 8, 11, 12): 0.0}
    for k, v in special.items():
        f[k] = v
    L.lbm_set_populations(lat.h, f)
    out = {}
    for dt in (torch.float32, torch.float64):
        t = torch.empty((2, 9, nz, nx), dtype=dt, device="cuda")
        torch.cuda.synchronize()
        L.lbm_export_state(lat.h, t)
        L.load().lbm_synchronize(lat.h)
        out[dt] = t.cpu().numpy()
    for k, v in special.items():
        assert np.array_equal(out[torch.float32][k], np.float32(v), equal_nan=True) or abs(out[torch.float32][k] - v) < 1e-7, k
    wide = out[torch.float64]  # the exact sums
    good = np.isfinite(wide)
    assert good.sum() == wide.size - 3
    # within half an ulp of them, and 2^-23 of that
    err = np.abs(out[torch.float32][good].astype(np.float64) - wide[good])
    assert np.all(err <= 0.5 * (1 + 2.0 ** -23) * np.spacing(np.abs(out[torch.float32][good])))
