"""GPU checks of a new context's node tile: where the rule leaves one tile an SM
(slabs of more than an SM's share of nodes, batches of mixed lengths, shared
memory for one CTA an SM only), a step's bits are those of any other tile."""
import numpy as np
import pytest

import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [ev.FP64, ev.FP32, ev.FP64_DF])
@pytest.mark.parametrize("lens,Q", [((9,), 8), ((5000,), 16), ((9731,), 32), ((12000,), 24), ((200,) * 24, 16),
                                    ((31, 700, 4001, 64) * 5, 20), ((333,) * 64, 8)])
def test_same_bits_as_another_tile(lens, Q, precision):
    sim = ev.Sim([ev.Params(nx=n, dx=0.25, Q=Q, precision=precision) for n in lens])
    nn = sum(lens)
    rng = np.random.default_rng(nn)
    n0 = 0.25 * (1 + 0.05 * rng.uniform(-1, 1, nn))
    assert 1 <= sim.tile_nodes() <= 64
    out = []
    for tile in (None, 7):
        if tile:
            sim.tune(tile)
        sim.init(n0, 0.05 * np.ones(nn), np.full(nn, 0.6))
        sim.step(2)
        out.append(sim.get_state())
    assert np.isfinite(out[0][0]).all()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    sim.close()


@pytest.mark.parametrize("Q", [17, 24, 32])
def test_sixteen_warps_where_a_tile_has_its_sm(Q):
    """1100 nodes in tiles of 11 and 64 (16 warps, one wave of CTAs on the SMs), 8 (8
    warps) and 1 (8 warps, several waves)."""
    nx = 1100
    sim = ev.Sim(ev.Params(nx=nx, dx=0.1, Q=Q, bc=ev.BC_OUTFLOW))
    rng = np.random.default_rng(Q)
    n0 = 0.25 * (1 + 0.3 * np.sin(np.arange(nx) / 40) + 0.02 * rng.uniform(-1, 1, nx))
    out = []
    for tile in (1, 8, 11, 64):
        sim.tune(tile)
        sim.init(n0, np.zeros(nx), np.full(nx, 0.6))
        sim.step(2)
        out.append(sim.get_state())
    assert np.isfinite(out[0][0]).all()
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0]) and np.array_equal(o[1], out[0][1])
    sim.close()
