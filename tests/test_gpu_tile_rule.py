"""The FP64 step on both sides of the grid size where its tiles go from 4 to 8
rows (456 tiles of 32 x 8), against the oracle; sizes, boundary kinds and
tolerance as in test_gpu_tiles.py."""
import numpy as np
import pytest
import torch

from oracle import dvbm_oracle as O
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


@pytest.mark.parametrize("Nx,Ny", [(608, 192), (607, 187), (609, 192), (97, 912), (97, 913)])
@pytest.mark.parametrize("lattice,kind", [(0, "periodic"), (0, "open"), (1, "open")])
def test_either_side_of_the_line(D, Nx, Ny, lattice, kind):
    F = I.random_smooth(Nx, Ny, seed=Nx + Ny, amp=0.1, Ma=0.4)
    dt = 0.3 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    mu = 8.0 * dt
    bcs, ob = None, None
    if kind == "open":
        bcs = [D.ZEROGRAD, D.ZEROGRAD, (D.WALL, (0.1, 0.0), 1.1), (D.WALL, (0.0, 0.0), 0.9)]
        ob = (O.BC(O.ZEROGRAD), O.BC(O.ZEROGRAD), O.BC(O.WALL, (0.1, 0.0), 1.1), O.BC(O.WALL, (0.0, 0.0), 0.9))
    sim = D.Simulation(Nx, Ny, 0.71, 1.4, mu, bcs=bcs, lattice=lattice, Lx=F.Lx, Ly=F.Ly, dt=dt)
    sim.init(*(torch.tensor(a) for a in (F.rho, F.ux, F.uy, F.T)))
    sim.step(2)
    s, _ = oracle_run(F, 0.71, 1.4, mu, dt, 2, bcs=ob, split="I" if lattice else "II")
    pops = sim.populations().cpu().numpy()
    perm = abi_to_oracle_perm(s.lat)
    n = s.lat.Q
    for a, b in ((pops[:n][perm], s.f.numpy()), (pops[n:][perm], s.g.numpy())):
        assert np.abs(a - b).max() < 1e-13 * np.abs(b).max()
