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
