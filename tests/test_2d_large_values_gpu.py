"""GPU check of the FP32 plane in a large unit of length: WENO-5 sums products of
four smoothness indicators and a difference, the ninth power of the differences of
F, which in FP32 ends near 5000.  Grid-scale noise of 4200 in F (a density of
11000 at sigma = 0.028) is within that, at the bar of the 2D model, 1e-5 of the
largest value of the right-hand side."""
import numpy as np
import pytest

import oracle as O
import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [(ev.FP32, 1e-5), (ev.FP64, 1e-11)])
def test_differences_near_the_end_of_the_float_range(prec, bar):
    nx, ny, Q, sigma = 40, 36, 4, 0.0281
    dx, n0 = sigma / 4, 0.25 / sigma ** 3
    sim = ev.Sim(ev.Params(nx=nx, ny=ny, dx=dx, Q=Q, dim=2, sigma=sigma, r_cut=6 * sigma, precision=prec))
    orc = O.Oracle2D(O.Setup2(nx=nx, ny=ny, Q=Q, dx=dx, dt=sim.dt(), sigma=sigma, rcut=6 * sigma))
    z = np.zeros((ny, nx))
    F, G = orc.equilibrium(z + n0, z, z, z + 0.6)
    noise = 1 + 0.9 * np.random.default_rng(1).uniform(-1, 1, F.shape)
    F, G = ((h * noise).astype(np.float32).astype(float) for h in (F, G))
    sim.set_state(F.ravel(), G.ravel())
    for got, want in zip(sim.rhs(), orc.rhs(F, G)):
        assert np.abs(got - want.ravel()).max() < bar * np.abs(want).max()
    sim.close()
