"""The scan of the initial fields (largest |u| + sqrt(gamma R T) for the CFL step,
largest pressure for the relaxation limit) in units where its single-precision
estimate underflows, 1e-13 to 1e-45 times the usual ones.  More cells than the
scan has threads (four blocks of 256 on each SM), smallest first, so that every
thread has to replace its first cell's maximum.

Tolerance: a speed is two products, a sum, two square roots and a sum, a pressure two
products, half an ulp each: 6 x 2^-53 < 1e-15 of it; 1e-14 and 1e-12 leave the reference its own."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
N = 512


@pytest.fixture(scope="module")
def D():
    import os
    from paper_2510_04197_gb300 import build, dvbm
    if not os.path.exists(dvbm.LIBPATH):
        build.build()
    assert torch.cuda.is_available()
    return dvbm


def _fields(speed, rho, T):
    """Speeds, temperature and density rise with the cell index by some 10 % in all."""
    s = 1.0 + 0.1 * np.arange(N * N).reshape(N, N) / (N * N)
    return rho * s, 0.3 * speed * s, 0.2 * speed * s, T * s


# unit of speed, of T (R = speed^2 / T) and of density; the usual units among them
@pytest.mark.parametrize("speed,T,rho", [(1.0, 1.0, 1.0), (1e-13, 1.0, 1.0), (1e-23, 1.0, 1.0), (1e-23, 1e-46, 1.0),
                                         (1e-20, 1e-30, 1e-30), (1.0, 1e-40, 1e-20), (1e10, 1.0, 1e-45),
                                         (1.0, 1e30, 1e-45), (1e25, 1e30, 1e5)])
def test_cfl_step_and_relaxation_limit(D, speed, T, rho):
    gamma, R = 1.4, speed ** 2 / T
    F = _fields(speed, rho, T)
    vmax = float((np.hypot(F[1], F[2]) + np.sqrt(gamma * R * F[3])).max())
    pmax = float((F[0] * R * F[3]).max())
    mu = pmax / (speed * N)  # relaxation time of about one cell's crossing
    kw = dict(R=R, T_ref=T, rho0=rho, T0=T, check_every=-1)
    dev = [torch.tensor(a, device="cuda") for a in F]
    with D.Simulation(N, N, 1.0, gamma, mu, cfl=0.01, **kw) as sim:
        sim.init(*dev)
        assert abs(sim.dt * vmax * N / 0.01 - 1.0) < 1e-14
    # a step at most the shortest relaxation time mu / pmax (a third of the fastest cell crossing)
    tau = 0.1 / (speed * N)
    mu = tau * pmax
    with D.Simulation(N, N, 1.0, gamma, mu, dt=tau * (1.0 - 1e-12), **kw) as sim:
        sim.init(*dev)
    with D.Simulation(N, N, 1.0, gamma, mu, dt=tau * (1.0 + 1e-12), **kw) as sim:
        with pytest.raises(D.DVBMError) as e:
            sim.init(*dev)
        assert e.value.status == D.EINVAL
