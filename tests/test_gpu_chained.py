"""Steps launched back to back against the same steps launched one at a time.

The short kernels of a step (low tiles, ghost layers, walls) start while their
predecessor runs and wait for it on the device: a value read too early would
differ.  The arithmetic is the same either way, so the populations are equal
bit for bit."""
import pytest
import torch

from paper_2510_04197_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    import os
    from paper_2510_04197_gb300 import build, dvbm
    if not os.path.exists(dvbm.LIBPATH):
        build.build()
    assert torch.cuda.is_available()
    return dvbm


# tiles of 2, 4 and 8 rows, ragged along both axes
@pytest.mark.parametrize("Nx,Ny", [(5, 7), (63, 61), (130, 75), (331, 97), (352, 385)])
@pytest.mark.parametrize("kind", ["periodic", "open"])
@pytest.mark.parametrize("lattice,storage", [(0, 0), (0, 1), (1, 0)])
def test_back_to_back_steps_equal_single_steps(D, Nx, Ny, kind, lattice, storage):
    F = I.random_smooth(Nx, Ny, seed=Nx, amp=0.1, Ma=0.4)
    dt = 0.1 * min(F.Lx / Nx, F.Ly / Ny) / 2.857
    bcs = None
    if kind == "open":
        bcs = [D.ZEROGRAD, D.ZEROGRAD, (D.WALL, (0.1, 0.0), 1.1), (D.WALL, (0.0, 0.0), 0.9)]
    out = []
    for single in (False, True):
        sim = D.Simulation(Nx, Ny, 0.71, 1.4, 8.0 * dt, bcs=bcs, lattice=lattice, storage=storage, Lx=F.Lx, Ly=F.Ly, dt=dt)
        sim.init(*(torch.tensor(a) for a in (F.rho, F.ux, F.uy, F.T)))
        if single:
            for _ in range(40):
                sim.step(1)
                torch.cuda.synchronize()
        else:
            sim.step(40)
        out.append(sim.populations().clone())
        sim.close()
    assert torch.equal(out[0], out[1])
