"""GPU checks of the 2D velocity kernels at the sizes where their tiles end:
the 32 x 32 advection tiles (an edge, one node beyond, grids narrower than
the stencil's halo), the 16-node collision groups (one group, a ragged last
group, an odd node count whose planes are not 16-byte aligned, more groups
than resident CTAs) and every order, whose matrices are compiled in; the WENO
regulariser below the flushing reciprocal's range; state copies on the device
against copies through the host.

One step from a non-equilibrium state against the oracle, at the bars of
the 2D model: FP64 1e-12 (step) and 1e-11 (right-hand side), FP32 1e-5 (Q^2-term
sums and WENO-5 in FP32, u = 2^-24)."""
import numpy as np
import pytest

import oracle as O
import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu

BAR = {ev.FP64: 1e-12, ev.FP32: 1e-5}


def rel(a, b):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())


def fields(nx, ny, seed):
    rng = np.random.default_rng(seed)
    x, y = np.meshgrid(np.arange(nx) / nx, np.arange(ny) / ny)
    n = 0.25 * (1 + 0.2 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y) + 0.02 * rng.uniform(-1, 1, (ny, nx)))
    return n, 0.03 * np.cos(2 * np.pi * y), 0.02 * np.sin(2 * np.pi * x), 0.6 * (1 + 0.03 * np.cos(2 * np.pi * (x + y)))


def case(nx, ny, Q, prec, eps=1e-6):
    sim = ev.Sim(ev.Params(nx=nx, dx=0.25, Q=Q, dim=2, ny=ny, precision=prec, weno_eps=eps))
    orc = O.Oracle2D(O.Setup2(nx=nx, ny=ny, Q=Q, dx=0.25, dt=sim.dt(), weno_eps=eps))
    F, G = orc.equilibrium(*fields(nx, ny, nx + ny))
    F, G = orc.step(F, G, 1)
    sim.set_state(F.ravel(), G.ravel())
    return sim, orc, F, G


@pytest.mark.parametrize("prec", [ev.FP64, ev.FP32])
@pytest.mark.parametrize("nx,ny,Q", [(8, 8, 4), (32, 32, 6), (33, 31, 10), (9, 65, 12), (64, 8, 14), (65, 41, 8)])
def test_step_at_tile_edges(nx, ny, Q, prec):
    sim, orc, F, G = case(nx, ny, Q, prec)
    sim.step(1)
    Fg, Gg = sim.state_2d()
    Fo, Go = orc.step(F, G, 1)
    assert rel(Fg, Fo) < BAR[prec] and rel(Gg, Go) < BAR[prec]
    sim.close()


@pytest.mark.parametrize("eps", [1e-10])
def test_small_weno_regulariser(eps):
    """eps below 1e-9: the WENO-5 divisors of flat regions are subnormal in
    FP32 (4 eps to the fourth power), so the kernel with the full quotient
    runs.  The oracle's step is well conditioned in eps where the state
    varies; the bar is the FP32 one."""
    sim, orc, F, G = case(24, 20, 6, ev.FP32, eps)
    sim.step(1)
    Fg, Gg = sim.state_2d()
    Fo, Go = orc.step(F, G, 1)
    assert np.all(np.isfinite(Fg)) and rel(Fg, Fo) < 1e-5 and rel(Gg, Go) < 1e-5
    sim.close()


@pytest.mark.parametrize("prec", [ev.FP64, ev.FP32])
def test_rhs_and_state_copies(prec):
    """The right-hand side (the advection kernel without its input term) and
    state copies with device arrays, equal to those through host arrays."""
    import torch
    sim, orc, F, G = case(19, 33, 8, prec)
    RF, RG = sim.rhs()
    RFo, RGo = orc.rhs(F, G)
    bar = 1e-11 if prec == ev.FP64 else 1e-4        # FP32: u times the size of h xi / dx over that of R
    assert rel(RF.reshape(RFo.shape), RFo) < bar and rel(RG.reshape(RGo.shape), RGo) < bar
    Fh, Gh = sim.get_state()
    Fd, Gd = sim.get_state(torch.empty(sim.NF, dtype=torch.float64, device="cuda"),
                           torch.empty(sim.NF, dtype=torch.float64, device="cuda"))
    assert np.array_equal(Fd.cpu().numpy(), Fh) and np.array_equal(Gd.cpu().numpy(), Gh)
    sim.step(1)
    a = sim.get_state()
    sim.set_state(Fd, Gd)
    sim.step(1)
    b = sim.get_state()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    sim.close()
