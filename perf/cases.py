"""What the speed of this framework is measured on: whole calls through its
public entry points, as the programs that use it make them.

Kinds of case
  slab    init + nsteps steps + state (and, FP64, moments): the 1D runs of
          phase separation, evaporation and planar interfaces
  batch   many independent slabs of uneven length and order in one context
  grad    forward and backward pass of EVRun (a density-profile loss)
  host    a host program that owns the state: upload, one step, moments
  plane   the two-dimensional model: init + nsteps steps + state

The state of an FP32 context holds 32-bit values; it is returned as such.

``exact`` evaluates the same method in 64-bit torch operations written out
from the equations (quadrature projections, textbook WENO-5, taps applied as
sums, reverse mode by autograd), sharing nothing with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

import paper_2503_15187_gb300 as ev
from paper_2503_15187_gb300.autograd import EVRun

F64 = torch.float64
PRECISION = {"fp64": ev.FP64, "fp32": ev.FP32, "fp64_df": ev.FP64_DF}

# vapour and liquid densities of the Maxwell construction at T / T_c (they
# depend on the ratio alone), and T_c of each model and spacing
COEXIST = ((0.60, 0.00588515230040, 0.77579276098354), (0.65, 0.01067016813555, 0.73020684580492),
           (0.70, 0.01775051174314, 0.68397971477169), (0.75, 0.02774277802527, 0.63644457181532),
           (0.80, 0.04148833882727, 0.58670053614258), (0.85, 0.06031675582287, 0.53335131263460),
           (0.90, 0.08674809830155, 0.47380599949925), (0.95, 0.12721884067666, 0.40155599024800))
T_C = {(1, "ev1", 0.1): 0.752953649962, (1, "ev1", 0.25): 0.755021457440, (1, "ev2", 0.1): 0.754629625070,
       (1, "ev2", 0.25): 0.754629625070, (2, "ev1", 0.25): 0.782364978542}


def listed():
    return [
        # the smallest run of phase separation: latency and launches count
        dict(name="separation_256_q16", kind="slab", nz=256, Q=16, dx=0.25, bc="periodic", force="ev1",
             precision="fp64", profile="noise", ratio=0.7, nbar=0.25, steps=40),
        # liquid-slab evaporation, the headline slab, plain FP64
        dict(name="evaporation_4096_q32", kind="slab", nz=4096, Q=32, dx=0.1, bc="outflow", force="ev1",
             precision="fp64", profile="liquid", ratio=0.8, nbar=0.0, steps=20),
        # its FP32 variant
        dict(name="evaporation_4096_q32_fp32", kind="slab", nz=4096, Q=32, dx=0.1, bc="outflow", force="ev1",
             precision="fp32", profile="liquid", ratio=0.8, nbar=0.0, steps=40),
        # its double-float variant, an odd length
        dict(name="evaporation_3001_q24_df", kind="slab", nz=3001, Q=24, dx=0.1, bc="outflow", force="ev1",
             precision="fp64_df", profile="liquid", ratio=0.75, nbar=0.0, steps=20),
        # the paper's planar interfaces held at a temperature, EV2 force
        dict(name="interface_2000_q16_ev2_iso", kind="slab", nz=2000, Q=16, dx=0.1, bc="periodic", force="ev2",
             precision="fp64", profile="pair", ratio=0.9, nbar=0.0, steps=30, dt=5e-3, iso=True),
        # 256 independent slabs, log-uniform lengths, mixed orders
        dict(name="batch_256", kind="batch", slabs=256, nz_min=128, nz_max=8192, steps=2, persistent=False),
        # a small batch, one persistent launch
        dict(name="batch_24_persistent", kind="batch", slabs=24, nz_min=100, nz_max=2000, steps=8, persistent=True),
        # calibration by gradients: forward and backward over checkpoints
        dict(name="calibration_1024_q24", kind="grad", nz=1024, Q=24, dx=0.25, ratio=0.75, nbar=0.25, steps=60,
             ckpt=20),
        # a host program that moves the state itself, every step
        dict(name="host_loop_4096_q32", kind="host", nz=4096, Q=32, dx=0.1, ratio=0.8),
        # 2D phase separation at its full size, a ragged middle size, a small one
        dict(name="plane_1024x1024_q16", kind="plane", nx=1024, ny=1024, Q=16, ratio=0.75, nbar=0.25, steps=2),
        dict(name="plane_333x250_q16", kind="plane", nx=333, ny=250, Q=16, ratio=0.75, nbar=0.25, steps=3),
        dict(name="plane_96x64_q8", kind="plane", nx=96, ny=64, Q=8, ratio=0.8, nbar=0.3, steps=10),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(("slab", "slab", "slab", "batch", "grad", "host", "plane", "plane", "plane"))
    ratio = round(rng.uniform(0.62, 0.94), 3)
    nbar = round(rng.uniform(0.15, 0.35), 3)
    if kind == "slab":
        force = rng.choice(("ev1", "ev1", "ev2"))
        iso = force == "ev2" and rng.random() < 0.5
        c = dict(kind=kind, nz=_log(rng, 64, 8192), Q=rng.choice((16, 16, 20, 23, 24, 32, 32)),
                 dx=rng.choice((0.1, 0.25)), bc="periodic" if iso else rng.choice(("periodic", "outflow")),
                 force=force, precision=rng.choice(("fp64", "fp64", "fp32", "fp64_df")),
                 profile=rng.choice(("noise", "liquid", "pair")), ratio=ratio, nbar=nbar, steps=rng.randint(4, 30),
                 iso=iso)
        if c["precision"] == "fp64_df":                              # whole groups of four orders
            c["Q"] -= c["Q"] % 4
        # the interface experiments run at the paper's spacing, step and order
        return dict(c, dx=0.1, dt=5e-3, Q=16) if iso else c
    if kind == "batch":
        return dict(kind=kind, slabs=_log(rng, 6, 128), nz_min=64, nz_max=_log(rng, 500, 8192),
                    steps=rng.randint(1, 4), persistent=rng.random() < 0.35)
    if kind == "grad":
        steps = rng.randint(6, 40)
        return dict(kind=kind, nz=_log(rng, 64, 2048), Q=rng.choice((16, 23, 24, 32)), dx=rng.choice((0.1, 0.25)),
                    ratio=ratio, nbar=nbar, steps=steps, ckpt=rng.randint(3, steps))
    if kind == "host":
        return dict(kind=kind, nz=_log(rng, 128, 8192), Q=rng.choice((16, 24, 32)), dx=rng.choice((0.1, 0.25)),
                    ratio=ratio)
    return dict(kind=kind, nx=_log(rng, 40, 1000), ny=_log(rng, 40, 1000), Q=rng.choice((8, 12, 16, 16)), ratio=ratio,
                nbar=nbar, steps=rng.randint(1, 2))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _t_c(c):
    return T_C[(2 if c["kind"] == "plane" else 1, c.get("force", "ev1"), c.get("dx", 0.25))]


def _temperature(c):
    return c["ratio"] * _t_c(c)


def _densities(ratio):
    t = np.array(COEXIST)
    return float(np.interp(ratio, t[:, 0], t[:, 1])), float(np.interp(ratio, t[:, 0], t[:, 2]))


def _profile(c, r):
    """Initial density of one slab: seeded noise about a mean, a liquid slab
    in its vapour, or a pair of planar interfaces."""
    nz, dx = c["nz"], c["dx"]
    kind = c.get("profile", "noise")
    if kind == "noise":
        return c["nbar"] * (1.0 + 0.01 * r.uniform(-1.0, 1.0, nz))
    n_v, n_l = _densities(c["ratio"])
    z = dx * (np.arange(nz) + 0.5) - 0.5 * nz * dx
    half = 0.25 * nz * dx if kind == "pair" else min(10.0, 0.2 * nz * dx)
    half *= r.uniform(0.9, 1.1)
    width = 2.0 if kind == "liquid" else math.sqrt(3.0 / (4.0 * math.pi * math.sqrt(3.0) * (1.0 - c["ratio"]) * _t_c(c)))
    n = n_v + 0.5 * (n_l - n_v) * (1.0 - np.tanh((np.abs(z) - half) / width))
    return n * (1.0 + 1e-4 * r.uniform(-1.0, 1.0, nz))


def _slab_params(c, **kw):
    return ev.Params(nx=c["nz"], dx=c["dx"], Q=c["Q"],
                     bc=ev.BC_OUTFLOW if c.get("bc") == "outflow" else ev.BC_PERIODIC,
                     precision=PRECISION[c.get("precision", "fp64")],
                     force_model=ev.EV2 if c.get("force") == "ev2" else ev.EV1, dt=c.get("dt", 0.0),
                     T_iso=_temperature(c) if c.get("iso") else 0.0, **kw)


def _batch(c, seed):
    """The slabs of a batch: lengths log-uniform, orders, T / T_c and mean
    densities uniform over their ranges, seeded noise.  Lengths and orders
    belong to the case, the rest to the seed."""
    shape, r = _rng(15187), _rng(seed)
    out = []
    for _ in range(c["slabs"]):
        nz = int(round(math.exp(shape.uniform(math.log(c["nz_min"]), math.log(c["nz_max"])))))
        s = dict(kind="slab", nz=nz, Q=int(shape.choice((16, 24, 32))), dx=0.25, bc="periodic", force="ev1",
                 ratio=float(r.uniform(0.6, 0.95)), nbar=float(r.uniform(0.15, 0.35)))
        out.append((s, _profile(s, r)))
    return out


def _plane_fields(c, seed):
    r = _rng(seed)
    ny, nx = c["ny"], c["nx"]
    x, y = np.arange(nx) / nx + r.uniform(), np.arange(ny)[:, None] / ny + r.uniform()
    n = c["nbar"] * (1.0 + 0.01 * r.uniform(-1.0, 1.0, (ny, nx)) + 0.05 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y))
    ux, uy = 0.03 * np.cos(2 * np.pi * y) + 0.0 * x, 0.02 * np.sin(2 * np.pi * x) + 0.0 * y
    T = _temperature(c) * (1.0 + 0.02 * np.cos(2 * np.pi * (x + y)))
    return n, ux, uy, T


def _host_fields(c, seed):
    """A slab with its liquid in the middle, in slow motion."""
    r = _rng(seed)
    n = _profile(dict(c, profile="liquid"), r)
    z = 2.0 * np.pi * (np.arange(c["nz"]) / c["nz"] + r.uniform())
    return n, 0.02 * np.sin(z), _temperature(c) * (1.0 + 0.01 * np.cos(2.0 * z))


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=F64, device="cuda")


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "grad":
        r = _rng(seed)
        n0 = _profile(c, r)
        return dict(case=c, params=_slab_params(c, ckpt_every=c["ckpt"]), phi=torch.tensor(1.0, dtype=F64),
                    T0=torch.tensor(_temperature(c), dtype=F64), n0=_dev(n0),
                    target=_dev(n0 * (1.0 + 0.02 * r.uniform(-1.0, 1.0, c["nz"]))))
    if kind == "host":
        n, u, T = _host_fields(c, seed)
        F, G = _equilibrium_1d(_Set(c["Q"]), _dev(n), _dev(u), _dev(T))
        pin = [torch.empty(c["Q"] * c["nz"], dtype=F64, pin_memory=True) for _ in range(2)]
        for p, h in zip(pin, (F, G)):
            p.copy_(h.reshape(-1))
        return dict(case=c, sim=ev.Sim(_slab_params(c)), pin=pin, F=pin[0].numpy(), G=pin[1].numpy())
    if kind == "plane":
        sim = ev.Sim(ev.Params(nx=c["nx"], ny=c["ny"], dx=0.25, Q=c["Q"], dim=2, precision=ev.FP32))
        n, ux, uy, T = _plane_fields(c, seed)
        fields = (_dev(n.ravel()), _dev(np.concatenate([ux.ravel(), uy.ravel()])), _dev(T.ravel()))
    elif kind == "batch":
        slabs = _batch(c, seed)
        sim = ev.Sim([_slab_params(s) for s, _ in slabs])
        if c["persistent"]:
            sim.set_persistent(True)
        n = np.concatenate([p for _, p in slabs])
        T = np.concatenate([np.full(s["nz"], _temperature(s)) for s, _ in slabs])
        fields = (_dev(n), _dev(np.zeros_like(n)), _dev(T))
    else:
        sim = ev.Sim(_slab_params(c))
        n = _profile(c, _rng(seed))
        fields = (_dev(n), _dev(np.zeros_like(n)), _dev(np.full(c["nz"], _temperature(c))))
    return dict(case=c, sim=sim, fields=fields, F=torch.empty(sim.NF, dtype=F64, device="cuda"),
                G=torch.empty(sim.NF, dtype=F64, device="cuda"))


def run(state):
    c = state["case"]
    if c["kind"] == "grad":
        leaf = [state[k].detach().requires_grad_() for k in ("phi", "T0", "n0")]
        n_end = EVRun.apply(*leaf, state["params"], c["steps"])
        ((n_end - state["target"]) ** 2).sum().backward()
        return dict(n=n_end.detach(), phi=leaf[0].grad, T0=leaf[1].grad, n0=leaf[2].grad)
    sim = state["sim"]
    if c["kind"] == "host":
        sim.set_state(state["F"], state["G"])
        sim.step(1)
        n, u, T, q, totals = sim.moments()
        return dict(n=n, u=u, T=T, q=q, totals=totals)
    sim.init(*state["fields"])
    sim.step(c["steps"])
    F, G = sim.get_state(state["F"], state["G"])
    if c["kind"] == "plane" or c.get("precision") == "fp32":
        return dict(F=F.float(), G=G.float())
    n, u, T, q, totals = sim.moments()
    return dict(F=F, G=G, n=n, u=u, T=T, q=q, totals=totals)


def work(case):
    """Bytes: inputs and outputs once, and, where the state is larger than the
    chip's caches, one read and one write of it per Runge-Kutta stage.
    Flops: the method's own count per node and velocity (WENO-5 faces of about
    60, Hermite transforms, collision and stage combination), two distributions."""
    c, kind = case, case["kind"]
    if kind == "plane":
        N, Q = c["nx"] * c["ny"], c["Q"]
        nv = N * Q * Q
        state = 8.0 * nv
        moved = 4 * 8.0 * N + state + (6 * c["steps"] * state if state > 120e6 else 0.0)
        return dict(bytes=moved, flops=3.0 * c["steps"] * nv * 2 * (120 + 4 * Q + 20))
    if kind == "batch":
        sizes = [(s["nz"], s["Q"]) for s, _ in _batch(c, 0)]
    else:
        sizes = [(c["nz"], c["Q"])]
    nodes, nv = sum(a for a, _ in sizes), sum(a * b for a, b in sizes)
    per = sum(a * b * 2.0 * (68 + 4 * b) for a, b in sizes)          # one right-hand side
    if kind == "host":
        return dict(bytes=16.0 * nv + 4 * 8.0 * nodes, flops=3 * per)
    if kind == "grad":                                               # reverse mode: twice the forward
        return dict(bytes=8.0 * nodes * 5, flops=9.0 * c["steps"] * per)
    size = 4 if c.get("precision") == "fp32" else 8
    return dict(bytes=3 * 8.0 * nodes + 2.0 * size * nv, flops=3.0 * c["steps"] * per)


# ---------------------------------------------------------------------------
# the method in 64-bit torch operations
# ---------------------------------------------------------------------------
class _Set:
    """Gauss-Hermite velocities, orthonormal Hermite polynomials on them
    (psi[l, k], l <= Q) and a quadrature of the local Gaussian."""

    def __init__(self, Q, nq=26):
        xi, w = np.polynomial.hermite_e.hermegauss(Q)
        z, wz = np.polynomial.hermite_e.hermegauss(nq)
        self.Q, self.xi, self.w = Q, _dev(xi), _dev(w / math.sqrt(2.0 * math.pi))
        self.z, self.wz = _dev(z), _dev(wz / math.sqrt(2.0 * math.pi))
        self.psi = torch.stack(self.hermite(self.xi, Q + 1))
        self.S = self.w[:, None] * self.psi[:Q].T                    # synthesis [k, l]
        r = torch.sqrt(torch.arange(1, Q + 1, dtype=F64, device="cuda"))
        # d/dxi on the set: (dh)_k = -w_k sum_{l<=Q-2} sqrt(l+1) psi_{l+1}(xi_k) sum_j psi_l(xi_j) h_j
        self.D = -(self.w[:, None] * (r[:, None] * self.psi[1:Q + 1]).T[:, :Q - 1]) @ self.psi[:Q - 1]

    def hermite(self, x, count):
        out = [torch.ones_like(x), x]
        for l in range(1, count - 1):
            out.append((x * out[l] - math.sqrt(l) * out[l - 1]) / math.sqrt(l + 1))
        return out[:count]

    def project(self, u, T, polys):
        """Coefficients E[poly(c) psi_l(u + c)], c ~ N(0, T): one [Q, ...] per poly."""
        acc = [0.0] * len(polys)
        for z, w in zip(self.z, self.wz):
            c = torch.sqrt(T) * z
            he = torch.stack(self.hermite(u + c, self.Q))
            for i, p in enumerate(polys):
                v = p(c)
                acc[i] = acc[i] + (w * v) * he
        return acc

    def project_1d(self, u, T, polys):
        """The same for one axis of nodes, the quadrature points as an array axis."""
        c = torch.sqrt(T) * self.z[:, None]
        he = torch.stack(self.hermite(u + c, self.Q))                # [Q, nq, nz]
        return [((self.wz[:, None] * p(c)) * he).sum(1) for p in polys]


def _weno(v0, v1, v2, v3, v4, eps=1e-6):
    q0 = (2 * v0 - 7 * v1 + 11 * v2) / 6
    q1 = (-v1 + 5 * v2 + 2 * v3) / 6
    q2 = (2 * v2 + 5 * v3 - v4) / 6
    b0 = 13 / 12 * (v0 - 2 * v1 + v2) ** 2 + 0.25 * (v0 - 4 * v1 + 3 * v2) ** 2
    b1 = 13 / 12 * (v1 - 2 * v2 + v3) ** 2 + 0.25 * (v1 - v3) ** 2
    b2 = 13 / 12 * (v2 - 2 * v3 + v4) ** 2 + 0.25 * (3 * v2 - 4 * v3 + v4) ** 2
    a0, a1, a2 = 0.1 / (eps + b0) ** 2, 0.6 / (eps + b1) ** 2, 0.3 / (eps + b2) ** 2
    return (a0 * q0 + a1 * q1 + a2 * q2) / (a0 + a1 + a2)


def _chi(n):
    eta = math.pi * n / 6
    return (2 - eta) / (2 * (1 - eta) ** 3)


def _transport(n, T, chi):
    """(rate 1/tau, Prandtl number, b n chi)."""
    bn = 2 * math.pi / 3 * n
    x = bn * chi
    k1, k2 = 4 / 25 * (1 + 12 / math.pi), 9 / 25 * (1 + 32 / (9 * math.pi))
    mu = 5 / 16 * torch.sqrt(T / math.pi) * (1 / chi + 0.8 * bn + k1 * bn * bn * chi)
    tau = mu / (n * T * (1 + 0.4 * x))
    pr = 2 / 3 * (1 + 0.6 * x) / (1 + 0.4 * x) * (1 + 0.8 * x + k1 * x * x) / (1 + 1.2 * x + k2 * x * x)
    return 1 / tau, pr, x


def _equilibrium_1d(s, n, u, T):
    F = s.S @ (n * s.project_1d(u, T, [lambda c: torch.ones_like(c)])[0])
    return F, T * F


class _Slab:
    """One slab in 64 bits: right-hand side and steps of the 1D model."""

    def __init__(self, c):
        self.s, self.c, self.dx = _Set(c["Q"]), c, c["dx"]
        self.dt = c.get("dt") or 0.5 * self.dx / float(self.s.xi[-1])
        self.T_iso = _temperature(c) if c.get("iso") else 0.0
        dx = self.dx
        simpson = lambda M: dx / 3 * np.array([1.0 if abs(j) == M else (4.0 if (j + M) % 2 else 2.0)  # noqa: E731
                                               for j in range(-M, M + 1)])
        m = round(1.0 / dx)
        z = dx * np.arange(-m, m + 1)
        self.fm = _dev(0.75 * simpson(m) * (1.0 - z * z))
        if c.get("force") == "ev2":
            a, kappa = 4 * math.pi / 3, 2 * math.pi / 15 * 6
            d1, d3 = np.array([1, -8, 0, 8, -1]) / (12 * dx), np.array([-1, 2, 0, -2, 1]) / (2 * dx ** 3)
            self.tap = _dev(2 * a * d1 + kappa * d3)
        else:
            M = round(6.0 / dx)
            z = dx * np.arange(-M, M + 1)
            az = np.maximum(np.abs(z), 1e-300)
            g = 2 * np.pi * np.where(np.arange(-M, M + 1) ** 2 < m * m, z, np.sign(z) * np.maximum(az, 0.5) ** -5.0)
            self.tap = _dev(simpson(M) * g)
        self.gi = {}

    def pad(self, f, h):
        if h not in self.gi:
            i = np.arange(-h, self.c["nz"] + h)
            i = np.clip(i, 0, self.c["nz"] - 1) if self.c.get("bc") == "outflow" else i % self.c["nz"]
            self.gi[h] = torch.as_tensor(i, device="cuda")
        return f[..., self.gi[h]]

    def taps(self, f, t):
        h = t.numel() // 2
        return self.pad(f, h).unfold(0, 2 * h + 1, 1) @ t

    def grad(self, f):
        p = self.pad(f, 2)
        return (p[:-4] - 8 * p[1:-3] + 8 * p[3:-1] - p[4:]) / (12 * self.dx)

    def moments(self, F, G):
        xi = self.s.xi[:, None]
        n = F.sum(0)
        u = (xi * F).sum(0) / n
        e = 0.5 * (xi - u) ** 2 * F + G
        return n, u, 2 * e.sum(0) / (3 * n), ((xi - u) * e).sum(0)

    def rhs(self, F, G, phi=1.0):
        s = self.s
        n, u, T, q = self.moments(F, G)
        chi = _chi(self.taps(n, self.fm))
        X = n * n * chi * T
        A, B, D = self.grad(X) / X, self.grad(T) / T, self.grad(u)
        force = phi * self.taps(n, self.tap)
        nu, pr, x = _transport(n, T, chi)
        sh = (1 - pr) * q / (n * T * T)
        polys = [lambda c: nu * (1 + sh * c * (c * c / (5 * T) - 0.6))
                 - x * (c * (A + 0.6 * (c * c / (2 * T) - 1.5) * B) + 0.4 * (1.5 * c * c / T - 1.5) * D),
                 lambda c: nu * T * (1 + sh * c * (c * c / (5 * T) - 0.2))
                 - x * (c * (T * A + 0.6 * (0.5 * c * c - 0.5 * T) * B) + 0.4 * (1.5 * c * c - 0.5 * T) * D)]
        out = []
        for h, a in zip((F, G), s.project_1d(u, T, polys)):
            p = self.pad(h, 3)
            nf = h.shape[-1] + 1
            v = [p[:, i:i + nf] for i in range(6)]
            face = torch.where(s.xi[:, None] > 0, _weno(*v[:5]), _weno(*v[:0:-1]))
            adv = -s.xi[:, None] * (face[:, 1:] - face[:, :-1]) / self.dx
            out.append(adv - force * (s.D @ h) - nu * h + s.S @ (n * a))
        return out

    def step(self, F, G, phi=1.0):
        L = lambda a, b: self.rhs(a, b, phi)  # noqa: E731
        dt = self.dt
        rF, rG = L(F, G)
        F1, G1 = F + dt * rF, G + dt * rG
        rF, rG = L(F1, G1)
        F2, G2 = 0.75 * F + 0.25 * (F1 + dt * rF), 0.75 * G + 0.25 * (G1 + dt * rG)
        rF, rG = L(F2, G2)
        F, G = F / 3 + 2 / 3 * (F2 + dt * rF), G / 3 + 2 / 3 * (G2 + dt * rG)
        if self.T_iso:
            n, u, T, _ = self.moments(F, G)
            a, b = (_equilibrium_1d(self.s, n, u, t) for t in (torch.full_like(T, self.T_iso), T))
            F, G = F + a[0] - b[0], G + a[1] - b[1]
        return F, G


class _Plane:
    """The two-dimensional model in 64 bits, one row of velocities at a time."""

    def __init__(self, c):
        self.s, self.dx = _Set(c["Q"], 16), 0.25
        self.dt = 0.5 * self.dx / (2 * float(self.s.xi[-1]))
        M, m, dx = round(6.0 / self.dx), math.ceil(1.0 / self.dx), self.dx
        x, w = np.polynomial.legendre.leggauss(48)
        self.force = []
        for a in range(-M, M + 1):
            for b in range(-M, M + 1):
                r = dx * math.hypot(a, b)
                if r == 0 or r > 6.0 + 1e-9:
                    continue
                end = 0.5 * math.pi if r >= 1.0 - 1e-12 else math.atan(r / math.sqrt(1.0 - r * r))
                J = 2 * r ** -7.0 * float((0.5 * end * w * np.sin(0.5 * end * (x + 1)) ** 6).sum())
                self.force.append((a, b, dx * dx * 6 * J * a * dx, dx * dx * 6 * J * b * dx))
        fm = [(a, b, 2 * math.sqrt(1.0 - dx * dx * (a * a + b * b))) for a in range(-m, m + 1) for b in range(-m, m + 1)
              if dx * dx * (a * a + b * b) < 1.0]
        total = sum(t[2] for t in fm)
        self.fm = [(a, b, v / total) for a, b, v in fm]

    @staticmethod
    def at(f, a, b):
        return torch.roll(f, (-b, -a), (-2, -1))

    def grad(self, f, ax):
        g = lambda j: torch.roll(f, -j, ax)  # noqa: E731
        return (g(-2) - 8 * g(-1) + 8 * g(1) - g(2)) / (12 * self.dx)

    def advect(self, h, v, ax):
        """-v dh/dx along axis ax of h [Q, ny, nx]; v [Q] or one value."""
        g = [torch.roll(h, -j, ax) for j in range(-2, 4)]            # nodes i-2 .. i+3
        face = torch.where(v > 0, _weno(*g[:5]), _weno(*g[:0:-1]))   # face i + 1/2
        return -v * (face - torch.roll(face, 1, ax)) / self.dx

    def fields(self, F, G):
        xi, Q = self.s.xi, self.s.Q
        n = F.sum((0, 1))
        ux = torch.tensordot(xi, F.sum(1), 1) / n
        uy = torch.tensordot(xi, F.sum(0), 1) / n
        e, qx, qy = torch.zeros_like(n), torch.zeros_like(n), torch.zeros_like(n)
        for i in range(Q):
            cx, cy = xi[i] - ux, xi[:, None, None] - uy
            k = 0.5 * (cx * cx + cy * cy) * F[i] + G[i]
            e, qx, qy = e + k.sum(0), qx + cx * k.sum(0), qy + (cy * k).sum(0)
        return n, ux, uy, 2 * e / (3 * n), qx, qy

    def rhs(self, F, G):
        s, Q = self.s, self.s.Q
        n, ux, uy, T, qx, qy = self.fields(F, G)
        nb = sum(w * self.at(n, a, b) for a, b, w in self.fm)
        chi = _chi(nb)
        fx, fy = torch.zeros_like(n), torch.zeros_like(n)
        for a, b, gx, gy in self.force:
            v = self.at(n, a, b)
            fx.add_(v, alpha=gx)
            fy.add_(v, alpha=gy)
        X = n * n * chi * T
        (Ax, Ay), (Bx, By) = ([self.grad(f, ax) / f for ax in (-1, -2)] for f in (X, T))
        Dxx, Dyx = self.grad(ux, -1), self.grad(ux, -2)
        Dxy, Dyy = self.grad(uy, -1), self.grad(uy, -2)
        nu, pr, x = _transport(n, T, chi)
        sq, dv = (1 - pr) / (n * T * T), Dxx + Dyy
        one = [(lambda c, a=a: c ** a) for a in range(4)]
        # one-axis syntheses of the local Gaussian times c^a, [4][Q, ny, nx]
        px, py = ([torch.tensordot(s.S, m, 1) for m in s.project(u, T, one)] for u in (ux, uy))
        # polynomials in (c_x, c_y) of nu f^S + J1 over F_MB, by powers (a, b)
        sx, sy = nu * sq * qx / (5 * T), nu * sq * qy / (5 * T)
        jF = {(0, 0): nu + 0.8 * x * dv, (1, 0): -4 * T * sx - x * (Ax - 1.2 * Bx), (0, 1): -4 * T * sy - x * (Ay - 1.2 * By),
              (2, 0): -0.4 * x * (Dxx + dv / 2) / T, (0, 2): -0.4 * x * (Dyy + dv / 2) / T, (1, 1): -0.4 * x * (Dxy + Dyx) / T,
              (3, 0): sx - 0.3 * x * Bx / T, (1, 2): sx - 0.3 * x * Bx / T, (0, 3): sy - 0.3 * x * By / T,
              (2, 1): sy - 0.3 * x * By / T}
        jG = {(0, 0): T / 2 * nu + 0.2 * x * T * dv, (1, 0): -T * T * sx - x * T / 2 * (Ax - 0.6 * Bx),
              (0, 1): -T * T * sy - x * T / 2 * (Ay - 0.6 * By), (2, 0): -0.2 * x * (Dxx + dv / 2),
              (0, 2): -0.2 * x * (Dyy + dv / 2), (1, 1): -0.2 * x * (Dxy + Dyx), (3, 0): T / 2 * sx - 0.15 * x * Bx,
              (1, 2): T / 2 * sx - 0.15 * x * Bx, (0, 3): T / 2 * sy - 0.15 * x * By, (2, 1): T / 2 * sy - 0.15 * x * By}
        out = []
        for h, poly in ((F, jF), (G, jG)):
            R = torch.empty_like(h)
            for i in range(Q):
                r = self.advect(h[i], s.xi[:, None, None], -2) + self.advect(h[i], s.xi[i], -1) - nu * h[i]
                r = r - fx * torch.tensordot(s.D[i], h, 1) - fy * torch.tensordot(s.D, h[i], 1)
                for b in range(4):
                    r = r + n * sum(px[a][i] * poly[a, b] for a in range(4 - b)) * py[b]
                R[i] = r
            out.append(R)
        return out

    def step(self, F, G):
        dt = self.dt
        rF, rG = self.rhs(F, G)
        F1, G1 = rF.mul_(dt).add_(F), rG.mul_(dt).add_(G)
        rF, rG = self.rhs(F1, G1)
        F2, G2 = (r.mul_(dt).add_(a).mul_(0.25).add_(b, alpha=0.75) for r, a, b in ((rF, F1, F), (rG, G1, G)))
        del F1, G1
        rF, rG = self.rhs(F2, G2)
        return tuple(r.mul_(dt).add_(a).mul_(2 / 3).add_(b, alpha=1 / 3) for r, a, b in ((rF, F2, F), (rG, G2, G)))

    def equilibrium(self, n, ux, uy, T):
        one = [lambda c: torch.ones_like(c)]
        px, py = (torch.tensordot(self.s.S, self.s.project(u, T, one)[0], 1) for u in (ux, uy))
        F = n * px[:, None] * py[None]
        return F, T / 2 * F


def _run_slab(c, n, u, T, steps):
    s = _Slab(c)
    F, G = _equilibrium_1d(s.s, n, u, T)
    for _ in range(steps):
        F, G = s.step(F, G)
    return F, G, s.moments(F, G)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "plane":
        p = _Plane(c)
        F, G = p.equilibrium(*(_dev(f) for f in _plane_fields(c, seed)))
        for _ in range(c["steps"]):
            F, G = p.step(F, G)
        return dict(F=F.reshape(-1), G=G.reshape(-1))
    if kind == "grad":
        s, r = _Slab(c), _rng(seed)
        n0 = _profile(c, r)
        target = _dev(n0 * (1.0 + 0.02 * r.uniform(-1.0, 1.0, c["nz"])))
        n0 = _dev(n0).requires_grad_()
        phi, T0 = (torch.tensor(v, dtype=F64, device="cuda", requires_grad=True) for v in (1.0, _temperature(c)))
        F, G = _equilibrium_1d(s.s, n0, torch.zeros_like(n0), T0 * torch.ones_like(n0))
        for _ in range(c["steps"]):
            # each step is formed again in the backward pass, so that the
            # graph of one step at a time is held
            F, G = torch.utils.checkpoint.checkpoint(s.step, F, G, phi, use_reentrant=False)
        n = F.sum(0)
        ((n - target) ** 2).sum().backward()
        return dict(n=n.detach(), phi=phi.grad, T0=T0.grad, n0=n0.grad)
    if kind == "host":
        _, _, (n, u, T, q) = _run_slab(c, *(_dev(f) for f in _host_fields(c, seed)), 1)
        return dict(n=n, u=u, T=T, q=q, totals=None)
    slabs = _batch(c, seed) if kind == "batch" else [(c, _profile(c, _rng(seed)))]
    got = []
    for s, n0 in slabs:
        n = _dev(n0)
        F, G, m = _run_slab(s, n, torch.zeros_like(n), torch.full_like(n, _temperature(s)), c["steps"])
        got.append((F.reshape(-1), G.reshape(-1)) + m)
    F, G, n, u, T, q = (torch.cat(v) for v in zip(*got))
    if c.get("precision") == "fp32":
        return dict(F=F, G=G)
    return dict(F=F, G=G, n=n, u=u, T=T, q=q, totals=None)
