"""What the FP64 step's arithmetic keeps of small values: the shared block exponent
of a tile against a strong density jump inside it, and the reciprocal's change of
method at 2^+-120.

The bound of one step from an equilibrium at rest: a tile's values are integers in
units of 2^-(58 - L) of its largest (L = ceil(log2 lq), beta = lp / lq; L = 0 for other
beta).  A face value has the truncation of its cell and, times at most beta, of the
smaller neighbouring difference, 1 + 2 x 2 units; two faces along each of two axes at
Courant numbers of at most 0.3: 6 units.  The flux sum and the dropped low products cut
four units of 2^-56 of the tile's largest.  Beside that 60 x 2^-53 of the largest
population of the cells that the update reads, for the roundings on either side
(test_gpu_tiles.py).  Twice this is allowed."""
import math

import numpy as np
import pytest
import torch
from scipy.ndimage import maximum_filter

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


# grids of 2-, 4- and 8-row tiles
@pytest.mark.parametrize("Nx,Ny,R", [(64, 64, 2), (128, 96, 4), (640, 192, 8)])
@pytest.mark.parametrize("beta,L", [(1.2, 3), (97.0 / 64.0, 6), (math.sqrt(2.0), 0)])
@pytest.mark.parametrize("lattice", [0, 1])
def test_a_density_ratio_of_a_million_in_a_tile(D, Nx, Ny, R, beta, L, lattice):
    F = I.random_smooth(Nx, Ny, seed=Nx, amp=0.1, Ma=0.2)
    x = np.arange(Nx)
    F.rho = F.rho * np.where((x % 32 >= 5) & (x % 32 < 20), 1.0, 1e-6)[None, :]
    F.ux, F.uy = 0.0 * F.ux, 0.0 * F.uy
    dt = 0.3 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    mu = 8.0 * dt
    sim = D.Simulation(Nx, Ny, 0.71, 1.4, mu, lattice=lattice, Lx=F.Lx, Ly=F.Ly, dt=dt, beta=beta, check_every=-1)
    sim.init(*(torch.tensor(a) for a in (F.rho, F.ux, F.uy, F.T)))
    sim.step(1)
    s, _ = oracle_run(F, 0.71, 1.4, mu, dt, 1, beta=beta, split="I" if lattice else "II")
    pops = sim.populations().cpu().numpy()
    perm = abi_to_oracle_perm(s.lat)
    n = s.lat.Q
    # before the step the largest population follows the density; the update reads two cells away
    for a, b in ((pops[:n][perm], s.f.numpy()), (pops[n:][perm], s.g.numpy())):
        size = np.maximum(np.abs(b).max(axis=0), F.rho * np.abs(b).max() / F.rho.max())
        near = maximum_filter(size, size=5, mode="wrap")
        tile = maximum_filter(size, size=(2 * R + 3, 2 * 32 + 3), mode="wrap")
        tol = 60 * 2.0 ** -53 * near + (6 * 2.0 ** -(58 - L) + 4 * 2.0 ** -56) * tile
        assert (np.abs(a - b) <= 2.0 * tol).all()


@pytest.mark.parametrize("k", [-130, -121, -120, -119, -1, 119, 120, 121, 130])
@pytest.mark.parametrize("lattice", [0, 1])
@pytest.mark.parametrize("Pr", [0.71, 2.0])
def test_density_scaled_by_a_power_of_two(D, k, lattice, Pr):
    """rho -> 2^k rho, mu -> 2^k mu scales every population by 2^k and leaves u and T
    alone.  All but 1/rho is exact under it; that is within one unit in the last place
    on either side of its range (the density is 0.8 to 1.25 times 2^k).  Five steps of
    about six roundings: 30 x 2^-53 of the largest population."""
    F = I.random_smooth(64, 48, seed=11, amp=0.1, Ma=0.4)
    dt = 0.3 * min(F.Lx / 64, F.Ly / 48) / 2.857
    out = []
    for e in (0, k):
        sim = D.Simulation(64, 48, Pr, 1.4, math.ldexp(8.0 * dt, e), lattice=lattice, Lx=F.Lx, Ly=F.Ly, dt=dt,
                           rho0=math.ldexp(1.0, e))
        sim.init(*(torch.tensor(a) for a in (np.ldexp(F.rho, e), F.ux, F.uy, F.T)))
        sim.step(5)
        out.append((np.ldexp(sim.populations().cpu().numpy(), -e), sim.moments()))
    (a, ma), (b, mb) = out
    n = len(a) // 2
    for s in (slice(0, n), slice(n, 2 * n)):
        assert np.abs(a[s] - b[s]).max() <= 30 * 2.0 ** -53 * np.abs(a[s]).max()
    for q in ("ux", "uy", "T"):
        assert float((ma[q] - mb[q]).abs().max()) <= 60 * 2.0 ** -53


@pytest.mark.parametrize("Nx,Ny", [(64, 64), (128, 96), (640, 192)])
@pytest.mark.parametrize("tiny", [-0.0, -1e-300, 1e-300, -3e-277])
def test_negligible_populations_stay_negligible(D, Nx, Ny, tiny):
    """gamma = 2 has no internal non-translational energy: g is zero.  Populations of g
    below every block's range, of either sign, leave f as it is and stay below 1e-270."""
    F = I.random_smooth(Nx, Ny, seed=5, amp=0.1, Ma=0.4)
    dt = 0.3 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    sim = D.Simulation(Nx, Ny, 0.71, 2.0, 8.0 * dt, Lx=F.Lx, Ly=F.Ly, dt=dt)
    sim.init(*(torch.tensor(a) for a in (F.rho, F.ux, F.uy, F.T)))
    st = sim.get_state()
    sim.step(4)
    clean = sim.populations().clone()
    assert float(clean[25:].abs().max()) < 1e-270
    sim.populations(st)[25:] = tiny
    sim.set_state(st)
    sim.step(4)
    got = sim.populations()
    assert torch.equal(got[:25], clean[:25])
    assert float(got[25:].abs().max()) < 1e-270
