"""GPU checks of the WENO-5 faces of an FP64 state beside a jump and over the
range of the regulariser: a flat side whose smoothness indicators stay at the
regulariser next to one at a jump, in both walk directions, from regularisers
that dominate every difference to ones far below the float range, and states
whose unit of length makes the densities large.

Tolerance: a face is a convex combination of values of the state to about
2^-45 of their differences; a step moves a value by at most half of the face
difference (CFL 0.5), so that the faces' part of the error stays below 1e-13 of
the largest value.  The bar is the FP64 bar against the oracle, 1e-12."""
import numpy as np
import pytest

import oracle as O
import paper_2503_15187_gb300 as ev

pytestmark = pytest.mark.gpu

EPS = (1e-6, 1e-14, 1e-18, 1e-20, 1e-24, 1e-32, 1e-40)


def rel(a, b):
    e = float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())
    return e if np.isfinite(e) else np.inf


def profile(kind, nx):
    """Densities of a slab of volume fraction up to 0.2 (sigma = 1)."""
    z = np.arange(nx) / nx
    if kind == "smooth":
        return 0.3 * (1 + 0.4 * np.sin(2 * np.pi * z) ** 3)
    if kind == "rough":                     # grid-scale noise
        return 0.3 * (1 + 0.3 * np.random.default_rng(nx).uniform(-1, 1, nx))
    n = np.full(nx, 0.1)
    if kind == "hat":                       # flat, up by a jump, flat, down again
        n[nx // 4:nx // 2] = 0.4
    elif kind == "spike":                   # a jump of one node on either side
        n[nx // 3] = 0.35
    else:                                   # jumps of many sizes between flat runs
        for i, j in enumerate((1e-1, 1e-3, 1e-5, 1e-7)):
            n[12 * i + 6:12 * i + 12] += j
    return n


def check(nx, Q, sigma, scale, eps, kind, precision):
    dx = 0.25 * sigma
    p = ev.Params(nx=nx, dx=dx, Q=Q, sigma=sigma, r_cut=6 * sigma, weno_eps=eps, precision=precision)
    sim = ev.Sim(p)
    orc = O.Oracle(O.Setup(nz=nx, Q=Q, dz=dx, dt=sim.dt(), sigma=sigma, rcut=6 * sigma, weno_eps=eps))
    n = scale * profile(kind, nx) / sigma ** 3
    F, G = orc.equilibrium(n, np.zeros(nx), np.full(nx, 0.65))
    sim.set_state(F.ravel(), G.ravel())
    R = sim.rhs()
    Ro = orc.rhs(F, G)
    top = [sim.dt() * float(np.abs(r - ro.ravel()).max()) / float(np.abs(h).max())
           for r, ro, h in zip(R, Ro, (F, G))]
    assert max(top) < 1e-12, top
    sim.step(1)
    Fg, Gg = sim.state_2d()
    Fo, Go = orc.step(F, G, 1)
    assert rel(Fg, Fo) < 1e-12 and rel(Gg, Go) < 1e-12
    sim.close()


@pytest.mark.parametrize("kind", ["hat", "spike", "jumps"])
@pytest.mark.parametrize("eps", EPS)
def test_jump_beside_flat(eps, kind):
    check(60, 16, 1.0, 1.0, eps, kind, ev.FP64)


@pytest.mark.parametrize("kind", ["smooth", "hat", "spike", "jumps"])
@pytest.mark.parametrize("eps", EPS)
def test_jump_beside_flat_double_float(eps, kind):
    """FP64_DF, whose faces do not scale their products."""
    check(60, 16, 1.0, 1.0, eps, kind, ev.FP64_DF)


@pytest.mark.parametrize("sigma", [1 / 512, 1 / 4096])
@pytest.mark.parametrize("kind", ["smooth", "hat", "spike"])
def test_small_unit_of_length(kind, sigma):
    """The same slab with lengths in a larger unit: densities of 4e7 and 2e10
    at the default regulariser."""
    check(60, 16, sigma, 1.0, 1e-6, kind, ev.FP64)


@pytest.mark.parametrize("scale", [1e-6, 1e-9, 1e-12])
@pytest.mark.parametrize("eps", EPS)
@pytest.mark.parametrize("kind", ["smooth", "rough"])
def test_small_differences(eps, scale, kind):
    """Rare gases: differences far below 1, with a regulariser above or below
    their squares."""
    check(60, 16, 1.0, scale, eps, kind, ev.FP64)
