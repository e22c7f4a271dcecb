"""GPU checks of 2D grids whose Fischer-Methfessel disc (the nodes within sigma)
holds thousands of taps beside a wide force disc: such grids are accepted up to
the size at which the staged densities of a tile alone fill the shared memory,
and the node fields do not depend on where the taps are read.

Tolerance: FP64 against the oracle 1e-12 of the largest value after a step; FP32
1e-5 (sums of thousands of FP32 terms, 2^-24 each, in the averages and forces)."""
import numpy as np
import pytest

import oracle as O
import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu


# (precision, sigma / dx, r_cut / sigma): the widest grids of each shape
@pytest.mark.parametrize("precision,m,rc", [(ev.FP32, 26, 4.0), (ev.FP32, 43, 2.5), (ev.FP32, 71, 1.5), (ev.FP32, 89, 1.2),
                                            (ev.FP64, 47, 1.5), (ev.FP64, 59, 1.2)])
def test_accepted(precision, m, rc):
    sim = ev.Sim(ev.Params(nx=16, ny=16, dx=1.0 / m, Q=4, dim=2, r_cut=rc, precision=precision))
    n = 0.25 * (1 + 0.01 * np.random.default_rng(m).uniform(-1, 1, 256))
    sim.init(n, np.zeros(512), np.full(256, 0.6))
    sim.step(1)
    F, G = sim.get_state()
    assert np.isfinite(F).all() and np.isfinite(G).all()
    sim.close()


@pytest.mark.parametrize("precision,m,rc,tol", [(ev.FP32, 43, 2.5, 1e-5), (ev.FP32, 8, 3.0, 1e-5), (ev.FP64, 40, 1.5, 1e-12),
                                                (ev.FP64, 8, 3.0, 1e-12)])
def test_against_oracle(precision, m, rc, tol):
    nx, ny, dx = 20, 18, 1.0 / m
    sim = ev.Sim(ev.Params(nx=nx, ny=ny, dx=dx, Q=4, dim=2, r_cut=rc, precision=precision))
    orc = O.Oracle2D(O.Setup2(nx=nx, ny=ny, Q=4, dx=dx, dt=sim.dt(), rcut=rc))
    rng = np.random.default_rng(m)
    n = 0.25 * (1 + 0.05 * rng.uniform(-1, 1, (ny, nx)))
    z = np.zeros((ny, nx))
    F, G = orc.equilibrium(n, z, z, z + 0.6)
    if precision == ev.FP32:
        F, G = F.astype(np.float32).astype(float), G.astype(np.float32).astype(float)
    sim.set_state(F.ravel(), G.ravel())
    sim.step(1)
    got = sim.get_state()
    for a, b in zip(got, orc.step(F, G, 1)):
        assert np.abs(a - b.ravel()).max() < tol * np.abs(b).max()
    sim.close()
