"""The 8-row kernels (grids beyond 456 tiles of 32 x 8) of every Prandtl branch and
limiter form, against the oracle: whole and ragged tiles, periodic and open, both
lattices, and the gradient whose recompute takes them.

Tolerances as derived in test_gpu_tiles.py (1e-13 of the largest population after two
steps) and test_gpu_adjoint_tiles.py (1e-12 of each field's largest gradient entry)."""
import math

import numpy as np
import pytest
import torch
from torch.utils.checkpoint import checkpoint

from oracle import dvbm_oracle as O
from paper_2510_04197_gb300 import autograd
from paper_2510_04197_gb300 import inputs as I
from helpers import abi_to_oracle_perm, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    import os
    from paper_2510_04197_gb300 import build, dvbm
    if not os.path.exists(dvbm.LIBPATH):
        build.build()
    assert torch.cuda.is_available()
    return dvbm


@pytest.mark.parametrize("Nx,Ny", [(640, 192), (609, 187)])
@pytest.mark.parametrize("kind", ["periodic", "open"])
@pytest.mark.parametrize("lattice,beta,Pr", [(0, 1.2, 0.71), (0, math.sqrt(2.0), 2.0), (0, 2.0, 1.0),
                                             (0, math.sqrt(3.0), 0.5), (1, 1.2, 2.0), (1, math.sqrt(2.0), 0.5),
                                             (1, 1.5, 1.0)])
def test_populations_match_the_oracle(D, Nx, Ny, kind, lattice, beta, Pr):
    F = I.random_smooth(Nx, Ny, seed=Nx + Ny, amp=0.1, Ma=0.4)
    dt = 0.3 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    mu = 8.0 * dt
    bcs, ob = None, None
    if kind == "open":
        bcs = [D.ZEROGRAD, D.ZEROGRAD, (D.WALL, (0.1, 0.0), 1.1), (D.WALL, (0.0, 0.0), 0.9)]
        ob = (O.BC(O.ZEROGRAD), O.BC(O.ZEROGRAD), O.BC(O.WALL, (0.1, 0.0), 1.1), O.BC(O.WALL, (0.0, 0.0), 0.9))
    sim = D.Simulation(Nx, Ny, Pr, 1.4, mu, bcs=bcs, lattice=lattice, Lx=F.Lx, Ly=F.Ly, dt=dt, beta=beta)
    sim.init(*(torch.tensor(a) for a in (F.rho, F.ux, F.uy, F.T)))
    sim.step(2)
    s, _ = oracle_run(F, Pr, 1.4, mu, dt, 2, bcs=ob, beta=beta, split="I" if lattice else "II")
    pops = sim.populations().cpu().numpy()
    perm = abi_to_oracle_perm(s.lat)
    n = s.lat.Q
    for a, b in ((pops[:n][perm], s.f.numpy()), (pops[n:][perm], s.g.numpy())):
        assert np.abs(a - b).max() < 1e-13 * np.abs(b).max()


@pytest.mark.parametrize("Pr,beta", [(2.0, 1.2), (1.0, 1.5), (0.71, math.sqrt(2.0))])
def test_gradients_match_the_oracle(D, Pr, beta):
    Nx, Ny, steps = 609, 187, 2
    F = I.random_smooth(Nx, Ny, seed=7, amp=0.08, Ma=0.4)
    dt = 0.2 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    mu = 8.0 * dt
    grads = []
    for dev in ("cuda", "cpu"):
        leaves = [torch.tensor(a, dtype=torch.float64, device=dev, requires_grad=True) for a in (F.rho, F.ux, F.uy, F.T)]
        if dev == "cuda":
            par = torch.tensor([mu, Pr, 1.4], dtype=torch.float64, requires_grad=True)
            rho, T = autograd.run(*leaves, par, steps, Lx=F.Lx, Ly=F.Ly, beta=beta, dt=dt)
        else:
            lat, P, grid = O.Lattice(), O.Params(Pr=Pr, gamma=1.4, mu=mu, beta=beta), O.Grid(Nx, Ny, F.Lx, F.Ly)
            f, g = O.init_populations(lat, P, *leaves)
            for _ in range(steps):
                f, g = checkpoint(lambda a, b: O.step(lat, P, grid, a, b, dt), f, g, use_reentrant=False)
            rho, _, _, T, _ = O.macroscopic(lat, P, f, g)
        (0.5 * ((rho - 0.9) ** 2 + (T - 1.2) ** 2).mean()).backward()
        grads.append([t.grad.cpu().numpy() for t in leaves])
    for a, b in zip(*grads):
        assert np.abs(a - b).max() < 1e-12 * np.abs(b).max()
