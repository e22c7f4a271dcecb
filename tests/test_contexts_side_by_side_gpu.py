"""GPU checks of contexts of different sizes in one process: the limit on a
kernel's dynamic shared memory belongs to the kernel, not to a context, so a
smaller context made later must not lower it under a larger one."""
import numpy as np
import pytest

import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu


def run(sim, n, T=0.6, steps=2):
    sim.init(n, np.zeros_like(n), np.full_like(n, T))
    sim.step(steps)
    out = [a.copy() for a in sim.get_state()]
    sim.rhs()
    sim.fields()
    return out


def noise(nx, seed):
    return 0.25 * (1 + 0.01 * np.random.default_rng(seed).uniform(-1, 1, nx))


# (order, spacing, tile of the first context; order and spacing of the second)
@pytest.mark.parametrize("Q,dx,tile,Q2,dx2", [(24, 0.1, 27, 12, 0.25), (20, 0.1, 24, 8, 0.25), (32, 0.1, 27, 4, 0.25),
                                              (32, 0.25, 64, 32, 0.25)])
@pytest.mark.parametrize("precision", [ev.FP64, ev.FP32, ev.FP64_DF])
def test_slabs(Q, dx, tile, Q2, dx2, precision):
    nx = 200
    n = noise(nx, 1)
    first = ev.Sim(ev.Params(nx=nx, dx=dx, Q=Q, precision=precision))
    first.tune(tile)
    alone = run(first, n)
    second = ev.Sim(ev.Params(nx=nx, dx=dx2, Q=Q2, precision=precision))
    small = run(second, n)
    beside = run(first, n)
    assert all(np.array_equal(a, b) for a, b in zip(alone, beside))
    assert all(np.array_equal(a, b) for a, b in zip(small, run(second, n)))
    first.close()
    second.close()


@pytest.mark.parametrize("persistent,T_iso", [(True, 0.0), (False, 0.6)])
def test_persistent_and_isothermal(persistent, T_iso):
    nx = 200
    n = noise(nx, 2)
    first = ev.Sim(ev.Params(nx=nx, dx=0.1, Q=32, T_iso=T_iso))
    first.tune(40)
    first.set_persistent(persistent)
    alone = run(first, n)
    second = ev.Sim(ev.Params(nx=nx, dx=0.25, Q=4, T_iso=T_iso))
    second.set_persistent(persistent)
    run(second, n)
    beside = run(first, n)
    assert all(np.array_equal(a, b) for a, b in zip(alone, beside))
    first.close()
    second.close()


def test_gradients():
    """The adjoint's kernels as well."""
    nx = 200
    n, bar = noise(nx, 3), np.random.default_rng(4).uniform(-1, 1, nx)

    def grad(Q, dx):
        sim = ev.Sim(ev.Params(nx=nx, dx=dx, Q=Q, ckpt_every=4))
        sim.init(n, np.zeros(nx), np.full(nx, 0.6))
        sim.step(4)
        return sim, sim.adjoint(bar)
    first, _ = grad(32, 0.1)
    second, _ = grad(4, 0.25)
    first.init(n, np.zeros(nx), np.full(nx, 0.6))
    first.step(4)
    first.adjoint(bar)
    first.close()
    second.close()


@pytest.mark.parametrize("precision", [ev.FP64, ev.FP32])
def test_planes(precision):
    """Two-dimensional contexts: a force disc of 40 nodes beside one of 12."""
    nx = ny = 48
    n = 0.25 * (1 + 0.01 * np.random.default_rng(5).uniform(-1, 1, nx * ny))
    z = np.zeros(2 * nx * ny)

    def go(sim):
        sim.init(n, z, np.full(nx * ny, 0.6))
        sim.step(1)
        out = [a.copy() for a in sim.get_state()]
        sim.rhs()
        return out
    first = ev.Sim(ev.Params(nx=nx, ny=ny, dx=0.15, Q=4, dim=2, precision=precision))
    alone = go(first)
    second = ev.Sim(ev.Params(nx=nx, ny=ny, dx=0.5, Q=4, dim=2, precision=precision))
    go(second)
    beside = go(first)
    assert all(np.array_equal(a, b) for a, b in zip(alone, beside))
    first.close()
    second.close()
