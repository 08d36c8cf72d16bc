"""Bands of a grid whose own size would take lower tiles than the whole grid's: the
tile height comes from the whole grid (dvbm_set_grid_rows), so bands of whole 8-row
tiles are bitwise the undecomposed run, forward and backward.

Tiles of 32 x 8 decide: the step takes 2 rows up to 38, 4 up to 456, the coded adjoint
step 4 up to 76."""
import pytest
import torch

from paper_2510_04197_gb300 import inputs as I

pytestmark = pytest.mark.gpu
FIELDS = ("rho0", "ux0", "uy0", "T0")


@pytest.fixture(scope="module")
def D():
    import os
    from paper_2510_04197_gb300 import build, dvbm
    if not os.path.exists(dvbm.LIBPATH):
        build.build()
    assert torch.cuda.is_available()
    return dvbm


def _pair(D, Nx, Ny, parts, every=0, steps=8, bcs=None, Pr=0.71, **kw):
    """The undecomposed run and the bands, both stepped."""
    from paper_2510_04197_gb300 import slab
    F = I.random_smooth(Nx, Ny, seed=Nx + Ny, amp=0.1, Ma=0.5)
    kw.update(Lx=F.Lx, Ly=F.Ly, dt=0.2 * min(F.Lx / Nx, F.Ly / Ny) / 2.857, check_every=-1)
    mu = 8.0 * kw["dt"]
    a = D.Simulation(Nx, Ny, Pr, 1.4, mu, bcs=bcs, **kw)
    b = slab.LocalSlabs(Nx, Ny, parts, Pr, 1.4, mu, bcs=bcs, **kw)
    assert all(h % 8 == 0 for h in b.heights[:-1])
    for s in (a, b):
        if every:
            s.record(every)
        s.init(*(torch.tensor(v, device="cuda") for v in (F.rho, F.ux, F.uy, F.T)))
        s.step(steps)
    return a, b


# whole grid 8 rows, bands 4 | 8 and 2 | 4 and 2, ragged upper band
@pytest.mark.parametrize("Nx,Ny,parts", [(512, 384, 2), (128, 920, 12), (128, 128, 2), (97, 131, 3)])
@pytest.mark.parametrize("lattice,kind", [(0, "periodic"), (0, "open"), (1, "periodic")])
def test_forward_bitwise(D, Nx, Ny, parts, lattice, kind):
    bcs = None if kind == "periodic" else [D.ZEROGRAD, D.ZEROGRAD, (D.WALL, (0.1, 0.0), 1.1), (D.WALL, (0.0, 0.0), 0.9)]
    a, b = _pair(D, Nx, Ny, parts, lattice=lattice, bcs=bcs)
    assert torch.equal(a.populations(), b.populations())


# adjoint step: whole grid 8 rows, bands 4 (forward step 4 and 4) | 8 and 8 (8 and 4) | 4 and 2 (4 and 2)
@pytest.mark.parametrize("Nx,Ny,parts,Pr", [(128, 192, 2, 0.71), (512, 384, 2, 2.0), (96, 160, 4, 1.0)])
def test_adjoint_bitwise(D, Nx, Ny, parts, Pr):
    a, b = _pair(D, Nx, Ny, parts, every=3, Pr=Pr)
    m = a.moments()
    dr, dT = (m["rho"] - 0.9) / m["rho"].numel(), (m["T"] - 1.1) / m["T"].numel()
    ga, gb = a.adjoint(dr, dT), b.adjoint(dr, dT)
    assert all(torch.equal(ga[k], gb[k]) for k in FIELDS)


def test_contract(D):
    F = I.random_smooth(32, 16, seed=2, amp=0.1, Ma=0.5)
    sim = D.Simulation(32, 16, 0.71, 1.4, 2e-3, dt=2e-4, Lx=F.Lx, Ly=F.Ly)
    for rows in (15, 2 ** 31 - 1):  # fewer than the context's own; out of range
        with pytest.raises(D.DVBMError) as e:
            sim.set_grid_rows(rows)
        assert e.value.status == D.EINVAL
    sim.set_grid_rows(4096).set_grid_rows(16)
    sim.record(2)
    sim.init(*(torch.tensor(v) for v in (F.rho, F.ux, F.uy, F.T)))
    sim.set_grid_rows(4096)
    sim.step(3)
    sim.set_grid_rows(4096)
    with pytest.raises(D.DVBMError) as e:  # the adjoint recomputes the steps with their tiles
        sim.set_grid_rows(16)
    assert e.value.status == D.ESTATE
