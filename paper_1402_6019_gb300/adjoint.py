"""Gradients of a run through the discrete adjoint of the step (library kernels).

A run is f_0 = W_l rho_init (the state lbm_set_fields makes with u = 0), then
f_{n+1} = S(f_n; theta) for `steps` steps, scored by the velocity / density profile objective
of lbm_adjoint_objective (targets of the kind Sec. IV measures: the x-averaged stream-flow
velocity and the density of species A across the lattice).  theta holds the NPARAM model
parameters in the order of the adjoint entry points:
G1 A, G1 B, G2 A, G2 B, G_AB, tau A, tau B, body_force.

The backward sweep needs every state f_n in reverse order.  Storing them all takes
steps x 9 ns nx nz values, so the forward keeps an exact snapshot every `checkpoint` steps and
the backward recomputes one segment at a time from its snapshot and sweeps it back
(lbm_adjoint_sweep): device memory for ceil(steps / checkpoint) snapshots and `checkpoint` recorded
states (twice that on small lattices where memory allows, the next segment recorded meanwhile), and
one extra forward run.

The adjoint runs in the lattice's precision unless told otherwise: an FP32 lattice records FP32
states and sweeps an FP32 adjoint; the parameter derivatives are accumulated in FP64 either way.
Every step, objective and adjoint step runs in the library; this module orders the calls and
holds the buffers.
"""
from __future__ import annotations

import torch

from . import lbm as L

NPARAM = 8
# Largest lattice whose backward sweep overlaps two segments: from there on a step's launches fill the
# GPU.  Gradients of two species, one buffer / two, us (20 steps a segment): FP32 256^2, 100 steps,
# 3,188 / 2,641; 384^2, 60 steps, 2,844 / 2,582; 512^2 3,776 / 3,720; 600^2, 40 steps, 3,493 / 3,497;
# FP64 256^2 16,209 / 15,352, 512^2 30,923 / 30,547.
OVERLAP_SITES = 512 * 512
_KEYS = [("G1", 0), ("G1", 1), ("G2", 0), ("G2", 1), ("G_AB", None), ("tau", 0), ("tau", 1), ("body_force", None)]


def theta_of(p: L.lbm_params) -> list:
    """The NPARAM parameters of p, in the adjoint's order."""
    return [getattr(p, k)[i] if i is not None else getattr(p, k) for k, i in _KEYS]


def set_theta(lat: L.Lattice, theta) -> None:
    """Write theta into the lattice's parameters (the other parameters are kept)."""
    p = lat.params
    for (k, i), v in zip(_KEYS, [float(t) for t in theta]):
        if i is None:
            setattr(p, k, v)
        else:
            getattr(p, k)[i] = v
    L.lbm_set_params(lat.h, p)


def _dtype(lat, dtype):
    if dtype is not None:
        return dtype
    return torch.float32 if lat.desc.precision == L.LBM_FP32 else torch.float64


def _device(lat):
    return torch.device("cuda", lat.desc.device)


def _handoff(device):
    """Wait for torch's work on its current stream: the library runs on the lattice's own
    stream, so tensors torch just wrote must be complete before the library reads them."""
    torch.cuda.current_stream(device).synchronize()


def overlaps(sites: int, segments: int, buffer_bytes: int, total_bytes: int, free_bytes) -> bool:
    """Whether a backward sweep takes a second buffer of a segment's states: where overlapping two
    segments pays, and the buffer is small beside the device's memory (1/64) or beside what is free of
    it (1/4; free_bytes: a function, asked only then: it costs 50 us of host time)."""
    if segments < 2 or sites > OVERLAP_SITES:
        return False
    return 64 * buffer_bytes <= total_bytes or 4 * buffer_bytes <= free_bytes()


class Run:
    """The forward run of a gradient: snapshots every `checkpoint` steps and the final state."""

    def __init__(self, lat: L.Lattice, rho_init: torch.Tensor, steps: int, checkpoint: int, dtype=None):
        if checkpoint < 1 or steps < 0:
            raise ValueError("checkpoint must be >= 1 and steps >= 0")
        self.lat, self.steps, self.checkpoint = lat, steps, checkpoint
        self.dtype = _dtype(lat, dtype)
        rho_init = rho_init.detach().contiguous()
        _handoff(_device(lat))
        lat.set_fields(rho_init)
        nb = L.lbm_snapshot_bytes(lat.h)
        self.snaps = []
        for k in range(0, steps, checkpoint):
            s = torch.empty(nb, dtype=torch.uint8, device=_device(lat))
            L.lbm_snapshot(lat.h, s)
            self.snaps.append(s)
            lat.step(min(checkpoint, steps - k))
        self.final = torch.empty((lat.ns, 9, lat.nz, lat.nx), dtype=self.dtype, device=_device(lat))
        L.lbm_export_state(lat.h, self.final)

    def objective(self, target_u, target_rho, grad=True):
        """(J as a 0-d FP64 device tensor, dJ/df_steps or None); synchronises."""
        J = torch.empty((), dtype=torch.float64, device=self.final.device)
        g = torch.empty_like(self.final) if grad else None
        target_u, target_rho = target_u.contiguous(), target_rho.contiguous()
        _handoff(self.final.device)
        L.lbm_adjoint_objective(self.lat.h, self.final, target_u, target_rho, J, g)
        self.lat.synchronize()
        return J, g

    def _second(self, seg: torch.Tensor):
        """A second buffer like seg (the next segment's states are recorded into it while one is swept
        back: the same results), or None."""
        total = torch.cuda.get_device_properties(seg.device).total_memory
        if not overlaps(self.lat.nx * self.lat.nz, len(self.snaps), seg.numel() * seg.element_size(), total,
                        lambda: torch.cuda.mem_get_info(seg.device)[0]):
            return None
        try:
            return torch.empty_like(seg)
        except torch.cuda.OutOfMemoryError:
            return None

    def backward(self, lam: torch.Tensor):
        """lam = dJ/df_steps; returns (dJ/drho_init [ns, nz, nx], dJ/dtheta [NPARAM]), FP64."""
        lat = self.lat
        lam = lam.to(self.dtype).contiguous().clone()
        grad = torch.zeros(NPARAM, dtype=torch.float64, device=lam.device)
        shape = (min(self.checkpoint, max(self.steps, 1)),) + tuple(lam.shape)
        seg = torch.empty(shape, dtype=self.dtype, device=lam.device)
        seg2 = self._second(seg)
        _handoff(lam.device)
        nsteps = [min(self.checkpoint, self.steps - k * self.checkpoint) for k in range(len(self.snaps))]
        try:
            L.lbm_adjoint_sweep(lat.h, self.snaps, nsteps, seg, seg2, lam, grad)
        except L.LbmError as e:  # the library's own buffers, allocated before lam and grad are touched, didn't fit
            if seg2 is None or e.code != L.LBM_ENOMEM:
                raise
            lat.synchronize()
            seg2 = None
            torch.cuda.empty_cache()
            L.lbm_adjoint_sweep(lat.h, self.snaps, nsteps, seg, None, lam, grad)
        g_rho = torch.empty((lat.ns, lat.nz, lat.nx), dtype=torch.float64, device=lam.device)
        L.lbm_adjoint_initial(lat.h, lam, g_rho)
        lat.synchronize()
        return g_rho, grad


def rollout_gradient(lat: L.Lattice, rho_init: torch.Tensor, steps: int, target_u: torch.Tensor,
                     target_rho: torch.Tensor, checkpoint: int = 25, dtype=None):
    """(J, dJ/drho_init [ns, nz, nx], dJ/dtheta [NPARAM]) of a run of `steps` steps."""
    run = Run(lat, rho_init, steps, checkpoint, dtype)
    J, lam = run.objective(target_u, target_rho)
    g_rho, grad = run.backward(lam)
    return float(J), g_rho, grad


def objective_value(lat: L.Lattice, rho_init: torch.Tensor, steps: int, target_u: torch.Tensor,
                    target_rho: torch.Tensor, dtype=None) -> float:
    """J of a run, without keeping snapshots or forming a gradient."""
    run = Run(lat, rho_init, steps, max(steps, 1), dtype)
    run.snaps = []
    return float(run.objective(target_u, target_rho, grad=False)[0])


class ProfileLoss(torch.autograd.Function):
    """J(rho_init, theta) of a run as a differentiable torch function.

    ProfileLoss.apply(lat, rho_init, theta, target_u, target_rho, steps, checkpoint): rho_init a
    CUDA float64 tensor [ns, nz, nx], theta a float64 tensor of NPARAM parameters (written into
    the lattice's parameters).  The backward pass recomputes the run from its snapshots and
    sweeps the adjoint, returning the gradients for rho_init and theta."""

    @staticmethod
    def forward(ctx, lat, rho_init, theta, target_u, target_rho, steps, checkpoint):
        set_theta(lat, theta.detach().cpu().tolist())
        run = Run(lat, rho_init, steps, checkpoint)
        J, lam = run.objective(target_u, target_rho)
        ctx.run, ctx.lam, ctx.theta_device = run, lam, theta.device
        return J

    @staticmethod
    def backward(ctx, gJ):
        g_rho, grad = ctx.run.backward(ctx.lam)
        ctx.run = ctx.lam = None
        return None, gJ * g_rho, (gJ * grad).to(ctx.theta_device), None, None, None, None
