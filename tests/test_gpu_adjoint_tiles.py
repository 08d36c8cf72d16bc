"""The adjoint step at the shapes where its tiles can go wrong, against the
oracle's discrete adjoint (torch.autograd on the oracle's forward map): tiles of
2, 4 and 8 rows, whole and ragged along each axis, one cell beyond a tile's edge,
the three Prandtl branches, the coded step (rational beta) and the general one.

Tolerance: each of four reverse steps rounds an entry about thirty times (the
projection, the pullback through the coefficients, the update) at the size of its
field's largest gradient entry: 4 x 30 x 2^-53 = 1.3e-14 of it, 1e-12 leaves two
orders.  The parameter gradients are sums of such terms of both signs over up to 1e5
cells and steps, which cancel by up to 1e4: 1e-8 relative."""
import math

import numpy as np
import pytest
import torch

from oracle import dvbm_oracle as O
from paper_2510_04197_gb300 import autograd
from paper_2510_04197_gb300 import inputs as I

pytestmark = pytest.mark.gpu
STEPS = 4


# tile height 2: up to 38 tiles of 32 x 8; 4: up to 76 (the recomputed forward step: 456); 8 above
@pytest.mark.parametrize("Nx,Ny", [(8, 8), (33, 9), (32, 130), (101, 75), (97, 160), (225, 73), (320, 70)])
@pytest.mark.parametrize("Pr,beta", [(0.71, 1.2), (2.0, 1.5), (1.0, 2.0), (0.5, math.sqrt(2.0))])
def test_gradients_match_the_oracle(Nx, Ny, Pr, beta):
    F = I.random_smooth(Nx, Ny, seed=Nx + Ny, amp=0.08, Ma=0.4)
    tgt = I.random_smooth(Nx, Ny, seed=99, amp=0.05, Ma=0.2)
    dt = 0.2 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    mu, gamma = 8.0 * dt, 1.4
    grads = []
    for dev in ("cuda", "cpu"):
        leaves = [torch.tensor(a, dtype=torch.float64, device=dev, requires_grad=True) for a in (F.rho, F.ux, F.uy, F.T)]
        rt, Tt = (torch.tensor(a, dtype=torch.float64, device=dev) for a in (tgt.rho, tgt.T))
        if dev == "cuda":
            par = torch.tensor([mu, Pr, gamma], dtype=torch.float64, requires_grad=True)
            rho, T = autograd.run(*leaves, par, STEPS, Lx=F.Lx, Ly=F.Ly, beta=beta, dt=dt)
        else:
            ps = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (mu, Pr, gamma)]
            P = O.Params(Pr=ps[1], gamma=ps[2], mu=ps[0], beta=beta)
            lat, grid = O.Lattice(), O.Grid(Nx, Ny, F.Lx, F.Ly)
            f, g = O.init_populations(lat, P, *leaves)
            for _ in range(STEPS):
                f, g = O.step(lat, P, grid, f, g, dt)
            rho, _, _, T, _ = O.macroscopic(lat, P, f, g)
        (0.5 * ((rho - rt) ** 2 + (T - Tt) ** 2).mean()).backward()
        params = par.grad.numpy() if dev == "cuda" else np.array([float(p.grad) for p in ps])
        grads.append(([t.grad.cpu().numpy() for t in leaves], params))
    (a, pa), (b, pb) = grads
    for x, y in zip(a, b):
        assert np.abs(x - y).max() < 1e-12 * np.abs(y).max()
    for k in range(3):
        if not (Pr == 1.0 and k == 1):  # one-sided at Pr = 1
            assert abs(pa[k] - pb[k]) < 1e-8 * abs(pb[k])
