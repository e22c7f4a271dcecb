"""GPU checks of the FP64 stage where its division of work changes: the node
work of a tile spread over warps and lanes (tiles of one node, of the sizes
at which a tap sum takes 8, 4, 2 and 1 lanes, and of more nodes than a warp
has lanes), the pool of face runs, and the WENO-5 faces' double-float part with
its range fallback.

Every per-node sum has a fixed order, so one step gives the same bits at
every tile; against the oracle it stays within the FP64 bar, 1e-12."""
import numpy as np
import pytest

import oracle as O
import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu

TILES = (1, 2, 3, 4, 5, 8, 9, 16, 17, 28, 29, 33, 64)


def rel(a, b):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())


def case(nx, Q, dx, bc, force, eps=1e-6, precision=ev.FP64):
    sim = ev.Sim(ev.Params(nx=nx, dx=dx, Q=Q, bc=bc, force_model=force, weno_eps=eps, precision=precision))
    orc = O.Oracle(O.Setup(nz=nx, Q=Q, dz=dx, dt=sim.dt(), bc=bc, force_model=force, weno_eps=eps))
    rng = np.random.default_rng(nx + Q)
    z = np.arange(nx) / nx
    n = 0.25 * (1 + 0.3 * np.tanh(8 * np.sin(2 * np.pi * z)) + 0.01 * rng.uniform(-1, 1, nx))
    F, G = orc.equilibrium(n, 0.03 * np.sin(2 * np.pi * z), 0.6 * (1 + 0.05 * np.cos(2 * np.pi * z)))
    return (sim, orc) + tuple(orc.step(F, G, 1))


@pytest.mark.parametrize("precision", [ev.FP64, ev.FP64_DF])
@pytest.mark.parametrize("nx,Q,dx,bc,force", [(70, 16, 0.25, ev.BC_PERIODIC, ev.EV1), (131, 24, 0.1, ev.BC_OUTFLOW, ev.EV1),
                                              (90, 32, 0.1, ev.BC_PERIODIC, ev.EV2)])
def test_same_bits_at_every_tile(nx, Q, dx, bc, force, precision):
    sim, orc, F, G = case(nx, Q, dx, bc, force, precision=precision)
    Fo, Go = orc.step(F, G, 1)
    ref = None
    for tile in TILES:
        sim.tune(tile)
        sim.set_state(F.ravel(), G.ravel())
        sim.step(1)
        Fg, Gg = sim.state_2d()
        if ref is None:
            assert rel(Fg, Fo) < 1e-12 and rel(Gg, Go) < 1e-12
            ref = Fg, Gg
        assert np.array_equal(Fg, ref[0]) and np.array_equal(Gg, ref[1]), tile
    sim.close()


@pytest.mark.parametrize("scale", [1.0, 1e-4])
@pytest.mark.parametrize("eps", [1e-2, 1e-14, 1e-29, 1e-40])
def test_face_range(eps, scale):
    """WENO regularisers from far above the differences to below the float
    range, where the faces of flat tail velocities take the FP64 form."""
    nx, Q, dx = 64, 16, 0.25
    sim = ev.Sim(ev.Params(nx=nx, dx=dx, Q=Q, weno_eps=eps))
    orc = O.Oracle(O.Setup(nz=nx, Q=Q, dz=dx, dt=sim.dt(), weno_eps=eps))
    z = np.arange(nx) / nx
    n = 0.3 * scale * (1 + 0.4 * np.sin(2 * np.pi * z) ** 3)
    F, G = orc.equilibrium(n, 0.05 * np.cos(2 * np.pi * z), 0.7 + 0 * z)
    sim.set_state(F.ravel(), G.ravel())
    sim.step(1)
    Fg, Gg = sim.state_2d()
    Fo, Go = orc.step(F, G, 1)
    assert rel(Fg, Fo) < 1e-12 and rel(Gg, Go) < 1e-12
    sim.close()
