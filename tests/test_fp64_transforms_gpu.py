"""GPU checks of the Hermite transforms of the FP64 stage, which run as plain
FP64 sums or as digit products on the tensor cores by Q (FP64_DF: always the
latter).

Tolerance: the digit products err by less than 2^-54 of a node's largest value
times the largest table entry, an FP64 sum of up to 16 terms by 16 times 2^-53 of
the same; either is far inside the FP64 bar against the oracle, 1e-12 after a
step, which the whole stage has to meet."""
import numpy as np
import pytest

import oracle as O
import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())


def fields(nx, seed):
    rng = np.random.default_rng(seed)
    z = np.arange(nx) / nx
    n = 0.25 * (1 + 0.5 * np.tanh(6 * np.sin(2 * np.pi * z)) + 0.02 * rng.uniform(-1, 1, nx))
    return n, 0.1 * np.sin(4 * np.pi * z), 0.6 * (1 + 0.2 * np.cos(2 * np.pi * z))


@pytest.mark.parametrize("precision", [ev.FP64, ev.FP64_DF])
@pytest.mark.parametrize("Q", list(range(4, 33)))
def test_every_order(Q, precision):
    """One step against the oracle at tiles that take one, a part of and several
    groups of eight nodes."""
    nx = 67
    sim = ev.Sim(ev.Params(nx=nx, dx=0.25, Q=Q, precision=precision))
    orc = O.Oracle(O.Setup(nz=nx, Q=Q, dz=0.25, dt=sim.dt()))
    F, G = orc.equilibrium(*fields(nx, Q))
    F, G = orc.step(F, G, 1)
    Fo, Go = orc.step(F, G, 1)
    ref = None
    for tile in (1, 7, 8, 30, 64):
        sim.tune(tile)
        sim.set_state(F.ravel(), G.ravel())
        sim.step(1)
        Fg, Gg = sim.state_2d()
        assert rel(Fg, Fo) < 1e-12 and rel(Gg, Go) < 1e-12, tile
        if ref is None:
            ref = Fg, Gg
        assert np.array_equal(Fg, ref[0]) and np.array_equal(Gg, ref[1]), tile
    sim.close()


@pytest.mark.parametrize("precision", [ev.FP64, ev.FP64_DF, ev.FP32])
def test_tables_outside_shared_memory(precision):
    """A tile of 64 nodes beside 1200 force taps to a side leaves no room for the
    stage's tables; tiles of 16 nodes hold them: the same bits."""
    nx, Q = 3000, 32
    sim = ev.Sim(ev.Params(nx=nx, dx=1 / 400, Q=Q, r_cut=3.0, precision=precision))
    F, G = O.Oracle(O.Setup(nz=64, Q=Q, dz=0.25, dt=1e-3)).equilibrium(*fields(64, 1))
    F, G = np.tile(F, 47)[:, :nx], np.tile(G, 47)[:, :nx]
    out = []
    for tile in (16, 64):
        sim.tune(tile)
        sim.set_state(np.ascontiguousarray(F).ravel(), np.ascontiguousarray(G).ravel())
        sim.step(1)
        out.append(sim.state_2d())
    assert np.isfinite(out[0][0]).all()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    sim.close()


@pytest.mark.parametrize("precision", [ev.FP64, ev.FP64_DF])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values_are_reported(bad, precision):
    nx, Q = 70, 32
    sim = ev.Sim(ev.Params(nx=nx, dx=0.25, Q=Q, precision=precision))
    F, G = O.Oracle(O.Setup(nz=nx, Q=Q, dz=0.25, dt=sim.dt())).equilibrium(*fields(nx, 3))
    F[Q - 1, 40] = bad
    with pytest.raises(ev.EvfdlbError):
        sim.set_state(F.ravel(), G.ravel())
        sim.step(1)
    sim.close()
