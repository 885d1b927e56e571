"""When a gradient's backward sweep takes a second buffer of states: never at the price of memory that a
gradient with one buffer would need."""
import numpy as np
import pytest
import torch

from paper_1402_6019_gb300 import adjoint as A
from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

GB = 1 << 30


@pytest.mark.parametrize("sites,segments,buffer,total,free,want", [
    (256 * 256, 8, 2 * GB, 280 * GB, 0, True),              # small beside the device
    (256 * 256, 1, 2 * GB, 280 * GB, 280 * GB, False),      # one segment: nothing to overlap
    (512 * 512, 2, 2 * GB, 280 * GB, 0, True),
    (512 * 512 + 1, 2, 2 * GB, 280 * GB, 280 * GB, False),  # a step's launches fill the GPU
    (512 * 512, 5, 38 * GB, 280 * GB, 100 * GB, False),     # 1000 two-species FP64 states a segment
    (512 * 512, 5, 38 * GB, 280 * GB, 200 * GB, True),
    (256 * 256, 2, 25 * GB, 280 * GB, 100 * GB, True),      # a quarter of what is free
    (256 * 256, 2, 25 * GB + 1, 280 * GB, 100 * GB, False),
])
def test_rule(sites, segments, buffer, total, free, want):
    assert A.overlaps(sites, segments, buffer, total, lambda: free) is want


@pytest.mark.gpu
def test_a_gradient_without_room_for_the_second_buffer_is_the_same(monkeypatch):
    """Where the memory is too full -- as reported, or refused by torch's allocator or by the library's --
    one buffer does, with the same bits."""
    nx, nz = 48, 40
    rho = torch.from_numpy(W.noise_field(nx, nz, seed=8, mean=0.7, amp=0.2, n_species=2)).cuda()
    tu = torch.zeros(nz, dtype=torch.float64, device="cuda")
    lat = L.Lattice(nx, nz, 2, L.LBM_FP64, L.LBM_PERIODIC, **dict(W.EMULSION_PARAMS, body_force=1e-5))
    swept = []
    sweep = L.lbm_adjoint_sweep

    def gradient(replace=None):
        def watched(h, snaps, nsteps, seg, seg2, lam, grad):
            swept.append(seg2 is not None)
            if seg2 is not None and replace == "library":
                raise L.LbmError(L.LBM_ENOMEM, "no memory")
            sweep(h, snaps, nsteps, seg, seg2, lam, grad)

        def refused(t, **kwargs):
            if t.dim() == 5:  # a segment's states
                raise torch.cuda.OutOfMemoryError("no memory")
            return torch.empty(t.shape, dtype=t.dtype, device=t.device)

        with monkeypatch.context() as m:
            m.setattr(L, "lbm_adjoint_sweep", watched)
            if replace == "reported":
                m.setattr(A, "overlaps", lambda *a: False)
            if replace == "torch":
                m.setattr(torch, "empty_like", refused)
            J, g_rho, theta = A.rollout_gradient(lat, rho, 14, tu, tu + 0.5, checkpoint=5)
        return np.concatenate([[J], g_rho.cpu().numpy().ravel(), theta.cpu().numpy()])

    want = gradient()
    assert swept == [True]
    for how, calls in (("reported", [False]), ("torch", [False]), ("library", [True, False])):
        swept.clear()
        assert np.array_equal(gradient(how), want), how
        assert swept == calls, how
