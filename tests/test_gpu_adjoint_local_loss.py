"""Gradients of losses on few cells, against the oracle's discrete adjoint.

The adjoint of a loss on one cell (a sensor, a mask) spreads two cells a step and
falls steeply towards its front, through every magnitude down to zero; a weighted
density loss hands the reverse pass such values at once, with exact zeros and both
signs beside them.  Tiles of 2, 4 and 8 rows.

Tolerance: a reverse step rounds the adjoint of each population about thirty times at
the size of the largest of them, and the gradient of every initial field is a sum of
them with factors of order one (a velocity's, where they nearly cancel at these short
time steps, carries the same absolute errors as the density's): 150 steps x 30 x 2^-53
= 5e-13 of the largest entry over the four fields at the worst, 1e-12."""
import math

import numpy as np
import pytest
import torch
from torch.utils.checkpoint import checkpoint

from oracle import dvbm_oracle as O
from paper_2510_04197_gb300 import autograd
from paper_2510_04197_gb300 import inputs as I

pytestmark = pytest.mark.gpu
# adjoint tiles of 2, 4 and 8 rows (up to 38, up to 76 and more tiles of 32 x 8)
SIZES = [(200, 8), (8, 320), (8, 640)]


def _gradients(dev, F, par, steps, dt, loss):
    """dL/d(rho, ux, uy, T) of the initial fields F on the GPU (the library) or the CPU (the oracle)."""
    leaves = [torch.tensor(a, dtype=torch.float64, device=dev, requires_grad=True) for a in (F.rho, F.ux, F.uy, F.T)]
    mu, Pr, gamma = par
    if dev == "cuda":
        p = torch.tensor(par, dtype=torch.float64, requires_grad=True)
        rho, T = autograd.run(*leaves, p, steps, Lx=F.Lx, Ly=F.Ly, dt=dt)
    else:
        Ny, Nx = F.rho.shape
        lat, P, grid = O.Lattice(), O.Params(Pr=Pr, gamma=gamma, mu=mu), O.Grid(Nx, Ny, F.Lx, F.Ly)
        f, g = O.init_populations(lat, P, *leaves)
        for _ in range(steps):
            f, g = checkpoint(lambda a, b: O.step(lat, P, grid, a, b, dt), f, g, use_reentrant=False)
        rho, _, _, T, _ = O.macroscopic(lat, P, f, g)
    loss(rho, T).backward()
    return [t.grad.cpu().numpy() for t in leaves]


def _compare(F, par, steps, dt, loss):
    got, ref = (_gradients(dev, F, par, steps, dt, loss) for dev in ("cuda", "cpu"))
    size = max(np.abs(b).max() for b in ref)
    for a, b in zip(got, ref):
        assert np.isfinite(a).all()
        assert np.abs(a - b).max() <= 1e-12 * size


@pytest.mark.parametrize("Nx,Ny", SIZES)
@pytest.mark.parametrize("Pr", [0.71, 1.0, 2.0])
def test_one_cell_loss_with_a_steep_front(Nx, Ny, Pr):
    """A time step of 1e-8 cell crossings: the front falls by about 1e9 a step and
    passes the smallest normal numbers within 40 steps."""
    F = I.random_smooth(Nx, Ny, seed=Nx + Ny, amp=0.08, Ma=0.4)
    dt = 1e-8 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    _compare(F, (100.0 * dt, Pr, 1.4), 40, dt, lambda rho, T: 0.5 * (rho[Ny // 2, Nx // 3] - 0.9) ** 2
             + 0.25 * (T[Ny // 2, Nx // 3] - 1.2) ** 2)


def test_one_cell_loss_at_the_default_time_step():
    """150 steps at the default CFL number 0.01 on 8 x 640 cells."""
    F = I.random_smooth(8, 640, seed=5, amp=0.08, Ma=0.4)
    h = min(F.Lx / 8, F.Ly / 640)
    dt = 0.01 * h / float((np.hypot(F.ux, F.uy) + np.sqrt(1.4 * F.T)).max())
    _compare(F, (2e-3, 0.71, 1.4), 150, dt, lambda rho, T: 0.5 * (rho[320, 3] - 0.9) ** 2)


@pytest.mark.parametrize("Nx,Ny", SIZES)
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_weights_through_the_smallest_numbers(Nx, Ny, sign):
    """A density weight exp(-(r / sigma)^2 / 2) that passes 1e-290, the subnormal
    numbers and zero, with no weight on T (g's adjoint starts from zeros of one sign)."""
    F = I.random_smooth(Nx, Ny, seed=Nx + Ny, amp=0.08, Ma=0.4)
    dt = 0.1 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    n = max(Nx, Ny)
    r = np.abs(np.arange(n) - n // 2)
    w1 = np.exp(-0.5 * (r / (n / 90.0)) ** 2)
    assert ((w1 > 0) & (w1 < 1e-290)).any() and (w1 == 0).any()
    w = torch.tensor(sign * (w1[None, :] if Nx == n else w1[:, None]) * np.ones((Ny, Nx)))
    _compare(F, (8.0 * dt, 0.71, 1.4), 3, dt, lambda rho, T: (w.to(rho.device) * rho).sum())
