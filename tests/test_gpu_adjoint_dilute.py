"""The FP64 adjoint step at densities far below rho0, at mixtures of small and ordinary pseudopotentials
(tiles that take the fixed-point sums beside tiles that don't) and at large densities, against torch's
own differentiation of the step in FP64 with -expm1 as psi (1 - exp, as the oracle has it, cancels there).

Bounds as for the adjoint step elsewhere: 1e-12 of max |lam|, parameter derivatives 1e-10 of their
value plus 1e-12 a site of the largest lam.  The couplings grow with rho0 as psi shrinks, so that
forces and derivatives keep their size and the bounds test psi's relative accuracy."""
import numpy as np
import pytest
import torch

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

pytestmark = pytest.mark.gpu

C = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))
WL = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
ATT, REP, BELT = {1: 4 / 15, 2: 1 / 10, 4: 1 / 120}, {1: 4 / 21, 2: 4 / 45, 4: 1 / 60, 5: 2 / 315, 8: 1 / 5040}, {1: 1 / 3, 2: 1 / 12}


def step(f, G1, G2, G_AB, tau, g, rho0, norm):
    at = lambda v, c: torch.roll(v, (-c[1], -c[0]), (-2, -1))  # v(x + c)
    col = lambda t: t.view(-1, 1, 1)
    rho = f.sum(1)
    jx, jz = [sum(f[:, l] * c[d] for l, c in enumerate(C) if c[d]) for d in (0, 1)]
    psi = -torch.expm1(-rho / col(rho0))
    F = [torch.zeros_like(rho), torch.zeros_like(rho)]
    for x in range(-2, 3):
        for z in range(-2, 3):
            q = x * x + z * z
            for d, e in ((0, x), (1, z)):
                if q and e:
                    F[d] = F[d] - psi * norm * (col(G1) * ATT.get(q, 0.0) + col(G2) * REP[q]) * e * at(psi, (x, z))
                    if f.shape[0] == 2 and q <= 2:
                        F[d] = F[d] - norm * G_AB * BELT[q] * e * rho * at(rho, (x, z)).flip(0)
    F[0] = F[0] + rho * g
    den = (rho / col(tau)).sum(0)
    u = [(j / col(tau)).sum(0) / den + col(tau) * w / rho for j, w in zip((jx, jz), F)]
    usq = u[0] ** 2 + u[1] ** 2
    out = []
    for l, c in enumerate(C):
        cu = c[0] * u[0] + c[1] * u[1]
        feq = WL[l] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq)
        out.append(torch.roll(f[:, l] - (f[:, l] - feq) / col(tau), (c[1], c[0]), (-2, -1)))
    return torch.stack(out, 1)


@pytest.mark.parametrize("ns", [1, 2])
@pytest.mark.parametrize("case", ["1e3", "1e8", "mixed", "vacuum", "dense"])
def test_adjoint_step_matches_torch(case, ns):
    nx, nz = 70, 9  # three tiles across, ragged; rows of two tiles and a half
    rng = np.random.default_rng(ns)
    rho = 0.7 + 0.3 * rng.uniform(-1, 1, (ns, nz, nx))
    scale = {"1e3": 1e3, "1e8": 1e8, "dense": 0.05}.get(case, 0.83)  # rho0
    if case in ("mixed", "vacuum"):  # psi of the right half below 2^-5
        rho[:, :, nx // 2:] *= 0.02 if case == "mixed" else 1e-6
    size = (scale / 0.83) ** 2 if scale > 1 else 1.0
    if case == "vacuum":
        size = 1e-3  # forces per density stay moderate beside a jump of 10^6
    G1, G2 = np.array([-9.0, -8.0]) * size, np.array([8.1, 7.1]) * size
    prm = dict(G1=tuple(G1), G2=tuple(G2), G_AB=0.3 if ns == 2 and case != "vacuum" else 0.0, tau=(0.8, 1.2), rho0=(scale,) * 2,
               weight_norm=1 / 3, body_force=1e-5)
    w = np.array(WL)[None, :, None, None]
    f = w * rho[:, None] * (1 + 0.05 * rng.uniform(-1, 1, (ns, 9, nz, nx)))
    lam_next = rng.standard_normal(f.shape)

    ft = torch.from_numpy(f).requires_grad_()
    par = [torch.tensor(v, dtype=torch.float64, requires_grad=True)
           for v in (prm["G1"][:ns], prm["G2"][:ns], prm["G_AB"], prm["tau"][:ns], prm["body_force"])]
    out = step(ft, par[0], par[1], par[2], par[3], par[4], torch.full((ns,), scale, dtype=torch.float64), 1 / 3)
    got = torch.autograd.grad((out * torch.from_numpy(lam_next)).sum(), [ft] + par, allow_unused=True)
    lam_ref = got[0].numpy()
    pad = lambda t: np.concatenate([t.numpy(), np.zeros(2 - ns)])
    grad_ref = np.concatenate([pad(got[1]), pad(got[2]), [0.0 if got[3] is None else float(got[3])], pad(got[4]), [float(got[5])]])

    lat = L.Lattice(nx, nz, ns, L.LBM_FP64, L.LBM_PERIODIC, **prm)
    d = [torch.from_numpy(a).cuda() for a in (f, lam_next)]
    lam, grad = torch.empty_like(d[0]), torch.zeros(8, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    L.lbm_adjoint_step(lat.h, d[0], d[1], lam, grad)
    lat.synchronize()
    err = np.abs(lam.cpu().numpy() - lam_ref).max() / np.abs(lam_ref).max()
    g = grad.cpu().numpy()
    print(case, ns, "lam", err, "theta", np.abs(g - grad_ref) / np.maximum(np.abs(grad_ref), 1e-300))
    assert err <= 1e-12
    # (a coupling's derivative shrinks as the coupling grows)
    atol = 1e-12 * nx * nz * np.abs(lam_next).max() * np.array([1 / size] * 4 + [1.0] * 4 if size > 1 else [1.0] * 8)
    assert np.all(np.abs(g - grad_ref) <= 1e-10 * np.abs(grad_ref) + atol), np.abs(g - grad_ref)
