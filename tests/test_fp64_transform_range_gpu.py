"""GPU checks of the digit products of the FP64 stage's Hermite transforms on
nodes whose coefficients do not decay as a Maxwellian's at rest near T = 1:
cold, hot and fast nodes, and slabs some hundred steps after a density step, whose
coefficients are near level in the order; and of non-finite values, which must
reach every velocity of their node and no node beyond the stencils.

Tolerances.  Right-hand side: the advection term |xi| / dx (h_{i+1/2} - h_{i-1/2})
of either side rounds four times, 2^-53 of the value each; the transforms have to
stay below that, 8 2^-53 max|xi| / dx of the largest value.  Step: the FP64 bar
against the oracle, 1e-12."""
import ctypes

import numpy as np
import pytest

import oracle as O
import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu


def setup(nx, Q, dx, **kw):
    sim = ev.Sim(ev.Params(nx=nx, dx=dx, Q=Q, **kw))
    return sim, O.Oracle(O.Setup(nz=nx, Q=Q, dz=dx, dt=sim.dt()))


def worst(got, want, like):
    return max(float(np.abs(g - w.ravel()).max() / np.abs(h).max()) for g, w, h in zip(got, want, like))


def flow(orc, nx, T, u):
    z = 2 * np.pi * np.arange(nx) / nx
    n = 0.3 * (1 + 0.3 * np.sin(z) + 0.01 * np.random.default_rng(nx).uniform(-1, 1, nx))
    return orc.equilibrium(n, u * (1 + 0.05 * np.cos(z)), T * (1 + 0.05 * np.sin(2 * z)))


@pytest.mark.parametrize("Q,T,u", [(Q, T, u) for Q in (17, 20, 24, 32) for T, u in ((0.15, 0.0), (0.3, 2.0), (0.6, 0.0), (1.0, 0.0))] +
                         [(24, 1.5, 1.0), (32, 1.5, 1.0)])
def test_cold_hot_and_fast_nodes(Q, T, u):
    nx, dx = 200, 0.25
    sim, orc = setup(nx, Q, dx)
    F, G = flow(orc, nx, T, u)
    sim.set_state(F.ravel(), G.ravel())
    assert worst(sim.rhs(), orc.rhs(F, G), (F, G)) < 8 * 2.0 ** -53 * orc.xi[-1] / dx
    sim.step(1)
    So = orc.step(F, G, 1)
    assert worst(sim.get_state(), So, So) < 1e-12
    sim.close()


def test_very_fast_nodes():
    nx, Q, dx = 200, 32, 0.25
    sim, orc = setup(nx, Q, dx)
    F, G = flow(orc, nx, 1.0, 4.0)
    sim.set_state(F.ravel(), G.ravel())
    sim.step(1)
    So = orc.step(F, G, 1)
    assert worst(sim.get_state(), So, So) < 1e-12
    sim.close()


@pytest.mark.parametrize("Q", [24, 32])
def test_after_a_density_step(Q):
    nx, dx = 256, 0.1
    sim, orc = setup(nx, Q, dx)
    z = dx * (np.arange(nx) + 0.5) - 0.5 * nx * dx
    F, G = orc.equilibrium(np.where(np.abs(z) < 0.2 * nx * dx, 0.58, 0.04), 0 * z, 0 * z + 0.7 * orc.critical_T())
    F, G = orc.step(F, G, 200)
    sim.set_state(F.ravel(), G.ravel())
    assert worst(sim.rhs(), orc.rhs(F, G), (F, G)) < 8 * 2.0 ** -53 * orc.xi[-1] / dx
    sim.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("node", [32, 39])
@pytest.mark.parametrize("Q,precision", [(17, ev.FP64), (32, ev.FP64), (16, ev.FP64_DF), (31, ev.FP64_DF)])
def test_non_finite_values_stay_with_their_node(Q, precision, node, bad):
    """dx = sigma and the merged stencil of EV2: no stencil is wider than three
    nodes, less than the eight that share a product."""
    nx = 70
    sim = ev.Sim(ev.Params(nx=nx, dx=1.0, Q=Q, precision=precision, force_model=ev.EV2))
    F, G = flow(O.Oracle(O.Setup(nz=nx, Q=Q, dz=1.0, dt=sim.dt())), nx, 0.6, 0.0)
    F[Q // 2 - 3, node] = bad
    sim.tune(64)
    sim.set_state(F.ravel(), G.ravel())
    out = [np.empty(nx * Q) for _ in range(2)]
    code = ev.lib().evfdlb_rhs(sim.h, ctypes.c_void_p(out[0].ctypes.data), ctypes.c_void_p(out[1].ctypes.data), 0)
    assert code != 0
    far = np.abs(np.arange(nx) - node) > 3
    for h in out:
        h = h.reshape(Q, nx)
        assert not np.isfinite(h[:, node]).any()
        assert np.isfinite(h[:, far]).all()
    sim.close()
