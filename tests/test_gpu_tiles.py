"""The tiled FP64 step against the oracle, population by population, at the
shapes where its tiles can go wrong: one cell beside and beyond a tile's edge
along each axis, the smallest grid, grids on both sides of the lines where the
tile height changes (2, 4 and 8 rows), every boundary kind, both limiter forms
and both lattices.

Tolerance: a step here rounds twice per population (the increment, the update)
on top of a block truncation of 2^-56 of the tile's largest value, the oracle
about ten times at the size of the largest population; 60 x 2^-53 = 7e-15 of it
after two steps.  1e-13 leaves an order of magnitude."""
import math

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


# tile height 2: up to 38 tiles of 32 x 8; 4: up to 76; 8 above
SIZES = [(4, 4), (31, 7), (32, 8), (33, 9), (64, 65), (200, 70), (193, 97), (289, 73), (321, 90)]


@pytest.mark.parametrize("Nx,Ny", SIZES)
@pytest.mark.parametrize("kind", ["periodic", "open"])
@pytest.mark.parametrize("lattice,beta,Pr", [(0, 1.2, 0.71), (0, math.sqrt(2.0), 2.0), (0, 2.0, 1.0), (1, 1.2, 2.0),
                                             (1, math.sqrt(2.0), 0.5)])
def test_tiles_match_the_oracle(D, Nx, Ny, kind, lattice, beta, Pr):
    F = I.random_smooth(Nx, Ny, seed=Nx + Ny, amp=0.1, Ma=0.4)
    # every population moves visibly, inside the step's limits (one cell, the relaxation time)
    dt = 0.3 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    mu = 8.0 * dt
    if kind == "periodic":
        bcs, ob = None, None
    else:
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


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_non_finite_cell_stays_within_its_stencil(D, value):
    """One population of one cell is not finite: the step reports it, and the
    cells that do not read it are as without it (they share its tile, whose
    block exponent leaves it out)."""
    F = I.random_smooth(96, 40, seed=3, amp=0.1, Ma=0.4)
    sim = D.Simulation(96, 40, 0.71, 1.4, 2e-3, Lx=F.Lx, Ly=F.Ly, dt=2e-4, check_every=-1)
    sim.init(*(torch.tensor(a) for a in (F.rho, F.ux, F.uy, F.T)))
    st = sim.get_state()
    sim.step(1)
    clean = sim.populations().clone()
    sim.populations(st)[8, 20, 40] = value
    sim.set_state(st)
    sim.step(1)
    got = sim.populations()
    keep = torch.ones(40, 96, dtype=torch.bool, device="cuda")
    keep[18:23, 40] = False
    keep[20, 38:43] = False
    assert float((got - clean)[:, keep].abs().max()) < 1e-13 * float(clean.abs().max())
    assert not torch.isfinite(got[:, 20, 40]).any()
    with pytest.raises(D.DVBMError):
        sim.totals()
