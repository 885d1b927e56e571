"""lbm_adjoint_sweep refuses two buffers of states that share memory (one is recorded while the other is
swept back), before anything is launched."""
import pytest
import torch

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_overlapping_buffers_are_refused(dtype):
    nx, nz, nsteps = 24, 17, [3, 2]
    lat = L.Lattice(nx, nz, 1, L.LBM_FP64, L.LBM_PERIODIC, **W.SINGLE_PARAMS)
    lat.set_fields(W.noise_field(nx, nz, seed=1))
    snaps = []
    for n in nsteps:
        s = torch.empty(L.lbm_snapshot_bytes(lat.h), dtype=torch.uint8, device="cuda")
        L.lbm_snapshot(lat.h, s)
        snaps.append(s)
        lat.step(n)
    m = 9 * nz * nx
    pool = torch.zeros(6 * m + 2, dtype=dtype, device="cuda")
    lam0 = torch.linspace(-1.0, 1.0, m, dtype=dtype, device="cuda").view(1, 9, nz, nx)
    lam, grad = lam0.clone(), torch.zeros(8, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    launches = L.lbm_launch_count(lat.h)
    for a, b in ((0, 0), (0, 1), (0, m), (0, 3 * m - 1), (3 * m - 1, 0), (2 * m, 0)):
        with pytest.raises(L.LbmError) as e:
            L.lbm_adjoint_sweep(lat.h, snaps, nsteps, pool[a:], pool[b:], lam, grad)
        assert e.value.code == L.LBM_EINVAL
    with pytest.raises(TypeError):  # of another type
        L.lbm_adjoint_sweep(lat.h, snaps, nsteps, pool[:3 * m], pool[3 * m:].to(torch.float16), lam, grad)
    with pytest.raises(ValueError):
        L.lbm_adjoint_sweep(lat.h, snaps, nsteps[:1], pool[:3 * m], None, lam, grad)
    assert L.lbm_launch_count(lat.h) == launches
    L.lbm_adjoint_sweep(lat.h, snaps, nsteps, pool, pool[3 * m:], lam, grad)  # side by side
    lat.synchronize()
    assert torch.isfinite(grad).all() and not torch.equal(lam, lam0)
