"""Workloads of the library as a user's program runs them, for timing.

listed() gives the fixed cases, draw(rng) one more of the same ranges,
prepare(case, seed) the simulation a program has in hand, run(state) one pass
through the public entry points, work(case) the bytes and operations a pass
cannot do without, and exact(case, seed) the same outputs in 64 bits from plain
torch (the method of arXiv 1710.09472 written out array by array, none of this
package's code).

Four kinds of pass:
  flow      n time steps of an isothermal box, then its density and current
            fields (every forward simulation: channel, shock tube, porous flow)
  gradient  forward and reverse sweep of the mean x-current through LBM.adjoint
  window    the same through torch.autograd (WindowCurrent), a design loop over
            the applied field
  thermal   n steps of the 1D thermal model, then its three fields
"""
from __future__ import annotations

import math

import numpy as np
import torch

THETA = 1.0 / 270.0  # the paper's electrons, with mu = 1
THERMAL_WEIGHT = ("mb", 1.0, 0.0)  # stable at every order of the thermal model

LATTICES = {"D2V9": (2, 9), "D3V19": (3, 19), "D3V27": (3, 27)}
BYTES = {"f32": 4, "f16": 2, "bf16": 2}


# ---------------------------------------------------------------------------
# The cases.
# ---------------------------------------------------------------------------
def _flow(name, vel, nx, ny, nz, storage, steps, walls, **over):
    case = dict(kind="flow", vel=vel, nx=nx, ny=ny, nz=nz, storage=storage, steps=steps, walls=walls, radius=6.0,
                porosity=0.7, tau=0.8, Ex=1e-6, Bz=0.0, force="term", local_mu=False)
    case.update(over)
    return case if name is None else dict(case, name=name)


def listed():
    return [
        # the smallest box anyone runs, the channel of the viscosity check: nothing but launches and latency
        _flow("poiseuille_32x64_f32", "D2V9", 32, 64, 1, "f32", 100, "channel"),
        # the closed shock tube: rows of 4096 cells, only eight of them, in bfloat16
        _flow("riemann_4096x8_bf16", "D2V9", 4096, 8, 1, "bf16", 100, "tube", tau=0.6, Ex=0.0),
        # the design loop: current through a 1024^2 sample, its gradient with respect to the field in every cell
        dict(name="window_1024x1024_f32", kind="window", vel="D2V9", nx=1024, ny=1024, nz=1, storage="f32", steps=100,
             window=25, every=20, walls="spheres", radius=8.0, porosity=0.6, tau=0.7, Ex=1e-6, Bz=1e-3, force="term"),
        # Ohm's law in a porous sample, the headline box: 16-bit storage, a magnetic field
        _flow("porous_256_f16", "D3V19", 256, 256, 256, "f16", 20, "spheres", Bz=1e-3),
        # the same in single precision, without the magnetic field
        _flow("porous_256_f32", "D3V19", 256, 256, 256, "f32", 10, "spheres", Ex=4e-6),
        # the gradient of the mean current of that sample with respect to the field in every cell
        dict(name="gradient_256_f16", kind="gradient", vel="D3V19", nx=256, ny=256, nz=256, storage="f16", steps=10,
             window=2, every=0, walls="spheres", radius=6.0, porosity=0.7, tau=0.8, Ex=1e-6, Bz=1e-3, force="term"),
        # the largest sample, 134 million cells
        _flow("porous_512_f16", "D3V19", 512, 512, 512, "f16", 4, "spheres", radius=10.0, porosity=0.65, Ex=2e-6,
              Bz=5e-4),
        # a scanned sample has the size it has: rows that are no whole number of 16 bytes
        _flow("porous_250x128x128_f16", "D3V19", 250, 128, 128, "f16", 20, "spheres", Bz=1e-3),
        # the 27-velocity lattice on the headline box
        _flow("porous_256_d3v27_f16", "D3V27", 256, 256, 256, "f16", 10, "spheres", Bz=1e-3),
        # every cell at the chemical potential of its own density
        _flow("porous_256_localmu_f16", "D3V19", 256, 256, 256, "f16", 10, "spheres", Bz=1e-3, local_mu=True),
        # heat pulses in one dimension, 16.8 million cells in 16 bits
        dict(name="thermal_16m_f16", kind="thermal", nx=1 << 24, storage="f16", steps=20, order=4, tau=0.8),
        # the same in single precision on a length that nothing divides
        dict(name="thermal_3m_f32", kind="thermal", nx=3000017, storage="f32", steps=20, order=4, tau=0.7),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi):
    """A box side: any integer half the time, else a multiple of 8, as chosen sizes are."""
    n = _log_uniform(rng, lo, hi)
    return n if rng.random() < 0.5 else max(8, n // 8 * 8)


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "flow", "gradient", "window", "thermal"])
    if kind == "thermal":
        return dict(kind="thermal", nx=_log_uniform(rng, 1 << 12, 1 << 24), storage=rng.choice(["f32", "f16", "bf16"]),
                    steps=20, order=rng.choice([3, 4, 4]), tau=rng.choice([0.7, 0.8]))
    porous = dict(walls="spheres", radius=rng.choice([3.0, 6.0, 8.0]), porosity=rng.choice([0.6, 0.7, 0.85]),
                  tau=rng.choice([0.7, 0.8, 0.9]), Ex=rng.choice([1e-6, 2e-6, 8e-6]), Bz=rng.choice([5e-4, 1e-3]),
                  force=rng.choice(["term", "shift"]))
    if kind == "window":
        steps = rng.choice([40, 60, 100])
        return dict(kind="window", vel="D2V9", nx=_side(rng, 64, 1024), ny=_side(rng, 64, 1024), nz=1,
                    storage=rng.choice(["f32", "f32", "f16"]), steps=steps, window=steps // 4,
                    every=rng.choice([0, 10, 20]), **porous)
    if kind == "gradient":
        vel = rng.choice(["D3V19", "D3V19", "D2V9"])
        d = LATTICES[vel][0]
        hi = 224 if d == 3 else 2048
        return dict(kind="gradient", vel=vel, nx=_side(rng, 24, hi), ny=_side(rng, 24, hi),
                    nz=_side(rng, 24, hi) if d == 3 else 1, storage=rng.choice(["f32", "f16"]), steps=10, window=2,
                    every=rng.choice([0, 4]), **porous)
    vel = rng.choice(["D2V9", "D3V19", "D3V19", "D3V27"])
    if vel == "D2V9":
        n = dict(nx=_side(rng, 32, 4096), ny=_side(rng, 8, 2048), nz=1)
    else:
        n = dict(nx=_side(rng, 24, 400), ny=_side(rng, 16, 256), nz=_side(rng, 16, 128))
    storage = rng.choice(["f32", "f16", "f16", "bf16"])
    steps = 20 if n["nx"] * n["ny"] * n["nz"] < 1 << 22 else 10
    return _flow(None, vel, n["nx"], n["ny"], n["nz"], storage, steps, **porous,
                 local_mu=vel == "D3V19" and rng.random() < 0.2)


# ---------------------------------------------------------------------------
# Inputs from the seed.
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _shape(case):
    """Array shape, x fastest: (ny, nx) or (nz, ny, nx)."""
    return (case["ny"], case["nx"]) if LATTICES[case["vel"]][0] == 2 else (case["nz"], case["ny"], case["nx"])


def _normal(shape, seed, k, std):
    g = torch.Generator(device=_device())
    g.manual_seed(1000003 * int(seed) + k)
    return torch.randn(shape, generator=g, device=_device(), dtype=torch.float32) * std


def _spheres(shape, radius, porosity, seed):
    """Overlapping disks or spheres (Boolean model): as many random centres as leave the porosity on average."""
    dev, d = _device(), len(shape)
    volume = math.pi * radius**2 if d == 2 else 4.0 / 3.0 * math.pi * radius**3
    count = max(1, round(-math.log(porosity) * math.prod(shape) / volume))
    centres = torch.from_numpy(np.random.RandomState(seed % (1 << 32)).rand(count, d) * np.array(shape)).to(dev)
    reach = torch.arange(-math.ceil(radius), math.ceil(radius) + 1, device=dev)
    ball = torch.stack(torch.meshgrid(*[reach] * d, indexing="ij"), -1).reshape(-1, d)
    mask = torch.zeros(math.prod(shape), dtype=torch.uint8, device=dev)
    size = torch.tensor(shape, device=dev)
    for part in centres.split(2048):
        cells = part.floor().long()[:, None, :] + ball[None]
        inside = (cells - part[:, None, :]).square().sum(-1) <= radius * radius
        cells = torch.remainder(cells, size)
        at = cells[..., 0]
        for k in range(1, d):
            at = at * shape[k] + cells[..., k]
        mask[at[inside]] = 1
    return mask.view(shape)


def _inputs(case, seed):
    """Solid cells, start density and velocity (xi units): the state a run has a while after its start, a density
    that varies by 0.1 % and a velocity of the size that the field drives."""
    shape = _shape(case)
    d = len(shape)
    rho = 1.0 + _normal(shape, seed, 1, 1e-3)
    u = _normal((d,) + shape, seed, 2, 1e-3)
    if case["walls"] == "channel":
        solid = torch.zeros(shape, dtype=torch.uint8, device=_device())
        solid[..., 0, :] = 1
        solid[..., -1, :] = 1
        y = torch.linspace(-1.0, 1.0, case["ny"], device=_device())
        u[0] += (3e-3 * (1.0 - y * y))[:, None]
    elif case["walls"] == "tube":
        solid = torch.zeros(shape, dtype=torch.uint8, device=_device())
        solid[..., 0] = 1
        solid[..., -1] = 1
        rho[..., : case["nx"] // 2] += 0.05
    else:
        solid = _spheres(shape, case["radius"], case["porosity"], seed)
    return solid, rho, u


def _field(case, seed):
    """Per-cell field E(x) of the design loop: N(Ex, Ex / 10) along x."""
    E = torch.zeros((2,) + _shape(case), dtype=torch.float32, device=_device())
    E[0] = case["Ex"] + _normal(_shape(case), seed, 3, 0.1 * case["Ex"])
    return E


def _thermal_inputs(case, seed):
    """Density, velocity and reduced temperature of the 1D box, relative to its weight's temperature."""
    n = (case["nx"],)
    return 1.0 + _normal(n, seed, 1, 5e-3), _normal(n, seed, 2, 1e-2), 1.0 + _normal(n, seed, 3, 5e-3)


# ---------------------------------------------------------------------------
# The simulation a program keeps, and one pass.
# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_1710_09472_gb300.lbm import LBM, Thermal

    dev = _device()
    if case["kind"] == "thermal":
        stat, theta, mu = THERMAL_WEIGHT
        sim = Thermal("D1V7", case["nx"], case["tau"], order=case["order"], storage=case["storage"], stat=stat,
                      theta=theta, mu=mu)
        rho, u, th = _thermal_inputs(case, seed)
        sim.init(rho, u, th * float(sim.const["thetabar_w"]))
        out = [torch.empty(case["nx"], dtype=torch.float32, device=dev) for _ in range(3)]
        return dict(case=case, sim=sim, out=out)
    dims = (case["nx"], case["ny"], case["nz"])[: LATTICES[case["vel"]][0]]
    solid, rho, u = _inputs(case, seed)
    sim = LBM(case["vel"], dims, case["tau"], E=(case["Ex"], 0.0, 0.0), B=(0.0, 0.0, case["Bz"]),
              storage=case["storage"], force=case["force"])
    sim.set_geometry(solid.reshape(-1))
    if case.get("local_mu"):
        sim.set_local_mu(True)
    sim.init_equilibrium(rho.reshape(-1), u.reshape(-1))
    state = dict(case=case, sim=sim)
    if case["kind"] == "flow":
        state["rho"] = torch.empty(sim.shape, dtype=torch.float32, device=dev)
        state["j"] = torch.empty((sim.D,) + sim.shape, dtype=torch.float32, device=dev)
    elif case["kind"] == "gradient":
        # loss: the x-current of the last steps, averaged over cells and steps
        state["w"] = torch.zeros((sim.D,) + sim.shape, dtype=torch.float32, device=dev)
        state["w"][0] = 1.0 / (sim.N * case["window"])
        state["dE"] = torch.empty((sim.D,) + sim.shape, dtype=torch.float64, device=dev)
    else:
        state["E"] = _field(case, seed).requires_grad_()
        state["B"] = torch.tensor([0.0, 0.0, case["Bz"]], device=dev, requires_grad=True)
        state["tau"] = torch.tensor(case["tau"], device=dev, requires_grad=True)
    return state


def run(state):
    case, sim = state["case"], state["sim"]
    steps = case["steps"]
    if case["kind"] == "flow":
        sim.step(steps)
        sim.moments(state["rho"], state["j"], totals=False)
        return {"rho": state["rho"], "j": state["j"]}
    if case["kind"] == "thermal":
        sim.step(steps)
        sim.moments(*state["out"], totals=False)
        return dict(zip(("rho", "j", "energy"), state["out"]))
    if case["kind"] == "gradient":
        got = sim.adjoint(steps - case["window"], steps, None, state["w"], case["every"], dL_dE=state["dE"])
        # the field is kept in FP32, so its optimiser takes the gradient in FP32 (as WindowCurrent hands it on)
        return {"loss": got["loss"], "dE": state["dE"].float(), "dB": got["dL_dB"].astype(np.float32),
                "dtau": got["dL_dtau"]}
    from paper_1710_09472_gb300.autograd import WindowCurrent

    totals = WindowCurrent.apply(state["E"], state["B"], state["tau"], sim, steps - case["window"], steps,
                                 case["every"])
    loss = totals[1] / (case["window"] * sim.N)
    dE, dB, dtau = torch.autograd.grad(loss, (state["E"], state["B"], state["tau"]))
    return {"totals": totals.detach(), "dE": dE, "dB": dB, "dtau": dtau}


def work(case):
    if case["kind"] == "thermal":
        q, n, b = 7, case["nx"], BYTES[case["storage"]]
        return {"bytes": case["steps"] * 2 * q * b * n + (q * b + 12) * n, "flops": case["steps"] * 30 * q * n}
    d, q = LATTICES[case["vel"]]
    n = case["nx"] * case["ny"] * case["nz"]
    b = BYTES[case["storage"]]
    fluid = n * {"spheres": case.get("porosity", 1.0), "channel": 1.0 - 2.0 / case["ny"],
                 "tube": 1.0 - 2.0 / case["nx"]}[case["walls"]]
    steps = case["steps"]
    if case["kind"] == "flow":  # each step reads and writes the populations; the fields read them once more
        return {"bytes": (steps * 2 + 1) * q * b * fluid + 4 * (1 + d) * n, "flops": steps * 13 * q * fluid}
    # a forward step, then a reverse step: the state read, the FP32 adjoint field read and written
    sweep = steps * (3 * q * b + 8 * q) * fluid + 4 * d * n
    if case["kind"] == "gradient":
        return {"bytes": sweep, "flops": steps * 40 * q * fluid}
    # through autograd the totals take a forward sweep of their own
    return {"bytes": sweep + steps * 2 * q * b * fluid + case["window"] * q * b * fluid,
            "flops": steps * 53 * q * fluid}


# ---------------------------------------------------------------------------
# The same in 64 bits: the paper's formulas on whole arrays.
# ---------------------------------------------------------------------------
def _weight_integrals(d, stat, theta, mu):
    """I_0, I_2, .. I_8 of the weight (Sec. 3), by Gauss-Legendre panels."""
    top = math.sqrt(1600.0 * theta) if stat == "mb" else math.sqrt(mu + 800.0 * theta)
    x, w = np.polynomial.legendre.leggauss(20)
    edges = np.linspace(0.0, top, 4001)
    h = 0.5 * np.diff(edges)
    xi = (0.5 * (edges[1:] + edges[:-1]))[:, None] + h[:, None] * x
    if stat == "mb":
        omega = (2 * math.pi * theta) ** (-0.5 * d) * np.exp(-0.5 * xi * xi / theta)
    else:
        omega = 1.0 / (np.exp(np.minimum((xi * xi - mu) / theta, 700.0)) + 1.0)
    return [math.pi ** (0.5 * d) / (2.0 ** (n - 1) * math.gamma(n + 0.5 * d))
            * float((h[:, None] * w * omega * xi ** (2 * n + d - 1)).sum()) for n in range(5)]


def _velocities(vel):
    d, q = LATTICES[vel]
    pairs = {"D2V9": [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)],
             "D3V19": [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1),
                       (0, 1, -1)]}
    pairs["D3V27"] = pairs["D3V19"] + [(1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)]
    e = [(0, 0, 0)]
    for v in pairs[vel]:
        e += [v, tuple(-c for c in v)]
    assert len(e) == q
    return e


class _Model:
    """The isothermal model of Sec. 9.1 with the forcing of Sec. 7, on lists of Q float64 arrays f_a."""

    def __init__(self, case, solid):
        self.case = case
        self.D, self.Q = LATTICES[case["vel"]]
        self.e = _velocities(case["vel"])
        self.I = _weight_integrals(self.D, "fd", THETA, 1.0)
        I0, I2, I4, I6 = self.I[:4]
        self.cs = math.sqrt(I2 / (3.0 * I4))
        J2 = I2 * I2 / (I4 * I0)
        shell = {"D2V9": [I0 * (1 - 5 * J2 / 9), I0 * J2 / 9, I0 * J2 / 36],
                 "D3V19": [I0 * (1 - 2 * J2 / 3), I0 * J2 / 18, I0 * J2 / 36],
                 "D3V27": [I0 - 2 * I2**2 / (3 * I4) - I6 * I2**3 / (27 * I4**3),
                           (3 * I2**2 * I4**2 + I6 * I2**3) / (54 * I4**3),
                           (3 * I4**2 * I2**2 - I6 * I2**3) / (108 * I4**3), I2**3 * I6 / (216 * I4**3)]}[case["vel"]]
        self.delta2 = 2.0 / ((self.D + 2) - J2 * self.D)  # Delta_2 squared
        self.w = [shell[sum(c * c for c in v)] for v in self.e]
        self.solid = solid.bool()
        self.axes = {0: -1, 1: -2, 2: -3}
        self.behind = [self.shift(self.solid, v) for v in self.e]  # x - e_a is solid
        self.tau = case["tau"]
        self.E = [case["Ex"], 0.0, 0.0]
        self.B = [0.0, 0.0, case["Bz"]]

    def shift(self, a, v):
        moves = [(v[k], self.axes[k]) for k in range(self.D) if v[k]]
        return torch.roll(a, [m[0] for m in moves], [m[1] for m in moves]) if moves else a

    @staticmethod
    def dot(v, a, scale=1.0):
        """scale v . a, leaving out zero components; 0.0 when none is left."""
        s = 0.0
        for c, x in zip(v, a):
            if c != 0 and not (isinstance(x, float) and x == 0.0):
                s = s + (c * scale) * x
        return s

    def equilibrium(self, a, rho, u, u2):
        """Sec. 5.1, Eq. feq-reduce-general-method-without-pol-eq."""
        I0, I2, I4 = self.I[:3]
        eu = self.dot(self.e[a], u, 1.0 / self.cs)
        return self.w[a] * rho * (1.0 / I0 + eu / I2 + eu * eu / (2 * I4) + self.k2(a) * u2)

    def k2(self, a):
        I0, I2, I4 = self.I[:3]
        xi2 = sum(c * c for c in self.e[a]) / self.cs**2
        return xi2 * (self.delta2 - 1) / (2 * self.D * I4) - I2 * self.delta2 / (2 * I0 * I4)

    def source(self, a, rho, u, uE):
        """S_a = (E + xi_a x B) . grad_u f^eq_a (Sec. 7, Eq. forcing-term-integrals-eq)."""
        _, I2, I4 = self.I[:3]
        xi = [c / self.cs for c in self.e[a]]
        eu, eE = self.dot(xi, u), self.dot(xi, self.E)
        B = self.B
        xB = [xi[1] * B[2] - xi[2] * B[1], xi[2] * B[0] - xi[0] * B[2], xi[0] * B[1] - xi[1] * B[0]]
        uxB = sum(u[d] * xB[d] for d in range(self.D))
        return self.w[a] * rho * (eE / I2 + eu * eE / I4 + 2 * self.k2(a) * (uE + uxB))

    def moments(self, f):
        rho = sum(f[1:], f[0])
        j = [sum(v[d] * f[a] for a, v in enumerate(self.e) if v[d]) / self.cs for d in range(self.D)]
        return rho, j

    def local_theta(self, rho):
        """thetabar(rho) - thetabar of the weight: I_2/I_0 at the chemical potential of the cell's density (Sec. 9.1;
        Sommerfeld series, exact to 1e-13 at these degenerate densities)."""
        def g(nu, eta):
            s, fall = 1.0, 1.0
            for k, zeta in enumerate((1.6449340668482264, 1.0823232337111382, 1.0173430619844491, 1.0040773561979443)):
                fall *= (nu - 2 * k) * (nu - 2 * k - 1)
                s = s + 2 * (1 - 2.0 ** (-1 - 2 * k)) * zeta * fall * eta ** (-2.0 * (k + 1))
            return eta**nu / math.gamma(nu + 1) * s

        nu, eta_w = 0.5 * self.D, 1.0 / THETA
        eta = eta_w * rho ** (1.0 / nu)
        for _ in range(6):  # g(eta) grows like eta^nu up to 1e-4: the fixed point gains four digits a turn
            eta = eta * (rho * g(nu, eta_w) / g(nu, eta)) ** (1.0 / nu)
        return 0.5 * THETA * (g(nu + 1, eta) / g(nu, eta) - g(nu + 1, eta_w) / g(nu, eta_w))

    def step(self, f):
        """Collide, then stream with halfway bounce-back; new arrays."""
        rho, j = self.moments(f)
        rho = torch.where(self.solid, torch.ones_like(rho), rho)
        u = [torch.where(self.solid, torch.zeros_like(x), x / rho) for x in j] + [0.0] * (3 - self.D)
        del j
        om = 1.0 / self.tau
        shift = self.case["force"] == "shift"
        if shift:
            E, B = self.E, self.B
            a = [E[0] + u[1] * B[2] - u[2] * B[1], E[1] + u[2] * B[0] - u[0] * B[2],
                 E[2] + u[0] * B[1] - u[1] * B[0]]
            u = [u[d] + self.tau * a[d] for d in range(self.D)] + [0.0] * (3 - self.D)
        u2 = sum(x * x for x in u[: self.D])
        uE = sum(u[d] * self.E[d] for d in range(self.D))
        extra = None
        if self.case.get("local_mu"):
            c2 = 1.0 / math.sqrt(self.I[2])
            d2 = math.sqrt(self.delta2)
            gg = c2 * d2
            cp = -c2 * self.I[1] / self.I[0] * d2
            extra = [0.5 * gg * (gg * sum(c * c for c in v) / self.cs**2 + self.D * cp) for v in self.e]
            dth = rho * self.local_theta(rho)
        post = []
        for a in range(self.Q):
            eq = self.equilibrium(a, rho, u, u2)
            if extra is not None:
                eq = eq + self.w[a] * extra[a] * dth
            v = f[a] + om * (eq - f[a])
            post.append(v if shift else v + self.source(a, rho, u, uE))
        out = []
        for a, v in enumerate(self.e):
            back = 0 if a == 0 else (a + 1 if a % 2 else a - 1)
            out.append(torch.where(self.behind[a], post[back], self.shift(post[a], v)))
        return out

    def start(self, rho, u):
        rho = rho.double()
        u = [x.double() for x in u] + [0.0] * (3 - self.D)
        u2 = sum(x * x for x in u[: self.D])
        return [self.equilibrium(a, rho, u, u2) for a in range(self.Q)]

    def fields(self, f):
        rho, j = self.moments(f)
        zero = torch.zeros_like(rho)
        return torch.where(self.solid, zero, rho), [torch.where(self.solid, zero, x) for x in j]


def _exact_thermal(case, seed):
    """The 1D thermal model: f^eq is the expansion of the shifted distribution on the weight's orthogonal polynomials up
    to the order (Sec. 4, Eq. feq-4order-01), written through the Gram matrix of the monomials; D1V7 of App. A."""
    stat, theta, mu = THERMAL_WEIGHT
    I = _weight_integrals(1, stat, theta, mu)
    even = [I[0], I[1], 3 * I[2], 15 * I[3], 105 * I[4]]  # integrals of the weight times xi^0, xi^2, .. xi^8
    roots = np.roots([105 * I[4], -210 * I[3], 147 * I[2], -36 * I[1]])
    x = max(r.real for r in roots if abs(r.imag) < 1e-9 and r.real > 0)
    e = np.array([0, 1, -1, 2, -2, 3, -3])
    half = np.linalg.solve(np.array([[float(s) ** (2 * k) if (s or k) else 1.0 for s in range(4)] for k in range(4)]),
                           [even[k] * x**k for k in range(4)])
    w = [half[0]] + [half[s] / 2 for s in (1, 1, 2, 2, 3, 3)]
    xi = e / math.sqrt(x)
    thw, g, order = I[1] / I[0], I[0] * I[2] / I[1] ** 2, case["order"]
    gram = np.array([[even[(i + k) // 2] if (i + k) % 2 == 0 else 0.0 for k in range(order + 1)]
                     for i in range(order + 1)])
    table = np.array([[c**k for k in range(order + 1)] for c in xi]) @ np.linalg.inv(gram) * np.array(w)[:, None]

    def equilibrium(rho, u, th):
        m = [rho, rho * u, rho * (th + u * u), rho * u * (3 * th + u * u),
             rho * (3 * g * th * th + 6 * th * u * u + u**4)][: order + 1]
        return [sum(table[a, k] * m[k] for k in range(order + 1)) for a in range(7)]

    rho, u, th = _thermal_inputs(case, seed)
    th = th * float(np.float64(thw))
    f = equilibrium(rho.double(), u.double(), th.double())
    om = 1.0 / case["tau"]

    def moments():
        return sum(f), sum(c * v for c, v in zip(xi, f)), sum(c * c * v for c, v in zip(xi, f))

    for _ in range(case["steps"]):
        r, j, en = moments()
        v = j / r
        eq = equilibrium(r, v, en / r - v * v)
        f = [torch.roll(f[a] + om * (eq[a] - f[a]), int(e[a])) for a in range(7)]
    return dict(zip(("rho", "j", "energy"), moments()))


def exact(case, seed):
    if case["kind"] == "thermal":
        return _exact_thermal(case, seed)
    solid, rho, u = _inputs(case, seed)
    m = _Model(case, solid)
    f = m.start(rho, u)
    del rho, u
    steps = case["steps"]
    if case["kind"] == "flow":
        with torch.no_grad():
            for _ in range(steps):
                f = m.step(f)
            r, j = m.fields(f)
            del f
            return {"rho": r, "j": torch.stack(j)}
    # the trajectory under autograd, each step recomputed in the reverse sweep
    from torch.utils.checkpoint import checkpoint

    n = solid.numel()
    if case["kind"] == "window":
        E = [x.double() for x in _field(case, seed)]
        m.tau = float(torch.tensor(case["tau"]))
        B = float(torch.tensor(case["Bz"]))
    else:
        E = [torch.full(_shape(case), case["Ex"] if d == 0 else 0.0, dtype=torch.float64, device=_device())
             for d in range(m.D)]
        B = case["Bz"]
    E = [x.requires_grad_() for x in E]
    B = [torch.tensor(v, dtype=torch.float64, device=_device(), requires_grad=True) for v in (0.0, 0.0, B)]
    tau = torch.tensor(m.tau, dtype=torch.float64, device=_device(), requires_grad=True)

    def one(tau, *rest):
        m.E = list(rest[: m.D]) + [0.0] * (3 - m.D)
        m.B = list(rest[m.D: m.D + 3])
        m.tau = tau
        return tuple(m.step(list(rest[m.D + 3:])))

    totals = torch.zeros(4, dtype=torch.float64, device=_device())
    for t in range(1, steps + 1):
        f = list(checkpoint(one, tau, *E, *B, *f, use_reentrant=False))
        if t > steps - case["window"]:
            r, j = m.fields(f)
            totals = totals + torch.stack([x.sum() for x in [r] + j + [torch.zeros_like(r)] * (3 - m.D)])
    loss = totals[1] / (case["window"] * n)
    got = torch.autograd.grad(loss, E + B + [tau], allow_unused=True)
    dE = torch.stack(got[: m.D])
    dB = torch.stack([torch.zeros_like(tau) if x is None else x for x in got[m.D: m.D + 3]])
    if m.D == 2:
        dB[:2] = 0.0  # only B_z acts in the plane
    if case["kind"] == "window":
        return {"totals": totals.detach(), "dE": dE, "dB": dB, "dtau": got[-1]}
    return {"loss": float(loss.detach()), "dE": dE, "dB": dB.cpu().numpy(), "dtau": float(got[-1])}
