"""Performance cases of the lattice library: the work a simulation has it do.

A lattice case is one segment of a run: the fields of a snapshot go into the lattice
(cl_set_state), a and a' are set (a' from Eq. Friedmann2), a number of time steps is
taken, and the updated fields and the volume-averaged energies come back.  The handle
(buffers, tiling, potential) is made once in prepare(), as a program keeps it over a run.
A surrogate case is one training step without the optimiser (forward, loss, backward, the
gradients), a spectrum case the measurement of the binned spectra of every field.

Models, couplings and lattice spacings are those of bench.py and the tests: lambda phi^4 in
conformal time, two-field preheating m2 phi^2 + g2 phi^2 chi^2, an axion with compact U(1)
links, ensembles of small lambda phi^4 lattices, the 3-48-48x4-2 convolution network.
"""
import math

import numpy as np
import torch

from paper_2607_24978_gb300 import cl

PREC = {"fp64": cl.CL_PREC_FP64, "fp32k": cl.CL_PREC_FP32_KAHAN, "fp32": cl.CL_PREC_FP32}
INTEG = {"vv2": cl.CL_INT_VV2, "yoshida4": cl.CL_INT_YOSHIDA4, "rk3-3": cl.CL_INT_RK3_3, "rk4-5": cl.CL_INT_RK4_5}
PASSES = {"vv2": 1, "yoshida4": 3, "rk3-3": 3, "rk4-5": 5}
ACT = {"relu": cl.CL_ACT_RELU, "gelu": cl.CL_ACT_GELU}

# the models: box side per site (dx), time step, alpha-time exponent, kappa
ONE = dict(dx=8.0 * math.pi / 32, dt=0.01, alpha=1.0, kappa=0.1)        # V = phi^4 / 4
TWO = dict(dx=8.0 * math.pi / 256, dt=0.005, alpha=0.0, kappa=0.1, g2=4e4)  # V = phi^2/2 + g2/2 phi^2 chi^2
U1 = dict(dx=2.0 * math.pi / 0.1 / 192, dt=0.01, alpha=0.0, kappa=1.0, alphaL=30.0, ws2=1e-4)  # V = phi^2 / 2


def _scalar(name, N, fields, precision, integrator, steps, gw=False):
    return dict(name=name, kind="scalar", N=N, fields=fields, precision=precision, integrator=integrator,
                steps=steps, gw=gw)


def _u1(name, N, precision, integrator, steps):
    return dict(name=name, kind="u1", N=N, precision=precision, integrator=integrator, steps=steps)


def listed():
    return [
        # the smallest run of the tests and the surrogate's training data: every launch counts
        _scalar("lphi4_32", 32, 1, "fp32k", "vv2", 200),
        # the headline: two-field preheating, one output interval
        _scalar("preheat_256", 256, 2, "fp32k", "yoshida4", 20),
        # the same model on a production-size lattice
        _scalar("preheat_512", 512, 2, "fp32k", "yoshida4", 10),
        # a lattice whose rows are no multiple of a vector (odd sizes symmetrise the Fourier grid)
        _scalar("preheat_odd_125", 125, 2, "fp32k", "yoshida4", 20),
        # double precision throughout: reference runs and precision studies
        _scalar("preheat_fp64_128", 128, 2, "fp64", "yoshida4", 10),
        # the non-symplectic evolver on the headline lattice
        _scalar("rk45_256", 256, 2, "fp32k", "rk4-5", 10),
        # gravitational waves sourced by the two fields
        _scalar("gw_256", 256, 2, "fp32k", "yoshida4", 10, gw=True),
        # axion inflation: Runge-Kutta steps of axion, links and electric field
        _u1("u1_rk33_192", 192, "fp32", "rk3-3", 10),
        # the same system with the leapfrog, on a size that the 32-site tiles do not divide
        _u1("u1_lf_100", 100, "fp32", "vv2", 20),
        # a parameter scan: many small lattices of three sizes advanced together, all read back
        dict(name="ensemble_256", kind="ensemble", members=256, sizes="32,48,64", steps=50),
        # one training step of the benchmark's network on the benchmark's lattice
        dict(name="surrogate_train_128", kind="surrogate", N=128, hidden=48, layers=6, activation="relu"),
        # a measurement: binned spectra of both fields and momenta
        dict(name="spectra_256", kind="spectra", N=256, fields=2, precision="fp32k"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """Any size of the range: multiples of 32 and of 4, even and odd ones."""
    n = _log_int(rng, lo, hi)
    m = rng.choice((1, 1, 2, 4, 8, 32))
    return min(hi, max(lo, (n + m // 2) // m * m))


def _steps(rng, sites, passes):
    """So many steps that a segment costs up to about 1.5e9 site passes, at most 200."""
    return max(1, min(200, int(rng.uniform(0.3, 1.0) * 1.5e9 / (sites * passes))))


def draw(rng):
    kind = rng.choice(("scalar", "scalar", "scalar", "scalar", "u1", "u1", "ensemble", "surrogate", "spectra"))
    if kind == "scalar":
        N = _size(rng, 16, 400)
        precision = rng.choice(("fp32k", "fp32k", "fp32k", "fp32", "fp64"))
        if precision == "fp64":
            N = min(N, 192)
        integrator = rng.choice(("vv2", "yoshida4", "yoshida4", "rk3-3", "rk4-5"))
        gw = integrator in ("vv2", "yoshida4") and precision != "fp64" and N <= 256 and rng.random() < 0.2
        c = _scalar("", N, rng.choice((1, 2)), precision, integrator,
                    _steps(rng, N ** 3 * (8 if precision == "fp64" else 1), PASSES[integrator]), gw)
    elif kind == "u1":
        N = _size(rng, 16, 192)
        precision = rng.choice(("fp32", "fp32", "fp64"))
        if precision == "fp64":
            N = min(N, 96)
        c = _u1("", N, precision, rng.choice(("vv2", "rk3-3", "rk4-5")),
                min(50, _steps(rng, N ** 3 * (32 if precision == "fp64" else 4), 5)))
    elif kind == "ensemble":
        members = _log_int(rng, 8, 256)
        c = dict(kind="ensemble", members=members,
                 sizes=rng.choice(("32,48,64", "32,48,64", "24,40,56", "16,32", "27,33,50", "64")),
                 steps=rng.randint(5, 50))
    elif kind == "surrogate":
        c = dict(kind="surrogate", N=16 * rng.randint(2, 8), hidden=rng.choice((16, 32, 48, 48)),
                 layers=rng.randint(3, 6), activation=rng.choice(("relu", "relu", "gelu")))
    else:
        c = dict(kind="spectra", N=_size(rng, 16, 256), fields=rng.choice((1, 2)),
                 precision=rng.choice(("fp32k", "fp32k", "fp64")))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _gen(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _dtype(precision):
    return torch.float64 if precision == "fp64" else torch.float32


def _noise(g, shape, mean, amp, dtype):
    return (mean + amp * torch.randn(shape, generator=g, device=_device(), dtype=torch.float32).double()).to(dtype)


def _scalar_inputs(N, fields, precision, seed):
    """Homogeneous values with white noise: phi (then chi) and their momenta."""
    g, dt, s = _gen(seed), _dtype(precision), (N, N, N)
    phi = [_noise(g, s, 1.0, 1e-2, dt)] + [_noise(g, s, 0.0, 1e-3, dt)] * (fields > 1)
    pi = [_noise(g, s, -0.1, 1e-2, dt)] + [_noise(g, s, 0.0, 1e-3, dt)] * (fields > 1)
    return phi, pi


def _u1_inputs(N, precision, seed):
    """The rolling axion, link angles and a divergence-free electric field (a backward curl)."""
    g, dt, s = _gen(seed), _dtype(precision), (N, N, N)
    phi, pi = _noise(g, s, 1.0, 1e-3, dt), _noise(g, s, -0.5, 1e-3, dt)
    theta = [_noise(g, s, 0.0, 1e-2, dt) for _ in range(3)]
    v = [_noise(g, s, 0.0, 5e-3, torch.float64) for _ in range(3)]
    back = lambda f, d: f - torch.roll(f, 1, 2 - d)  # noqa: E731
    E = [(back(v[(i + 2) % 3], (i + 1) % 3) - back(v[(i + 1) % 3], (i + 2) % 3)).to(dt).contiguous() for i in range(3)]
    return phi, pi, theta, E


def _ensemble_sizes(case):
    sizes = [int(x) for x in case["sizes"].split(",")]
    r = np.random.default_rng(1234)
    return [int(x) for x in r.choice(sizes, case["members"])]


def _ensemble_inputs(case, seed):
    """Members back to back: phi and pi of each, its fluctuations of a size of its own."""
    g, sizes = _gen(seed), _ensemble_sizes(case)
    V = [n ** 3 for n in sizes]
    amp = torch.repeat_interleave(
        10.0 ** (-3.0 + 1.5 * torch.rand(len(V), generator=g, device=_device())),
        torch.tensor(V, device=_device()))
    phi = 1.0 + amp * torch.randn(sum(V), generator=g, device=_device())
    pi = amp * torch.randn(sum(V), generator=g, device=_device())
    return sizes, phi, pi


def _surrogate_inputs(case, seed):
    """Normalised (phi, pi, a) and the target state; He-scaled weights."""
    g, N = _gen(seed), case["N"]
    x = torch.randn((N, N, N, 3), generator=g, device=_device())
    x[..., 2] = 0.5
    target = (x[..., :2] + 0.3 * torch.randn((N, N, N, 2), generator=g, device=_device())).contiguous()
    r = np.random.default_rng(int(seed))
    h, L = case["hidden"], case["layers"]
    shapes = [(h if l else 3, 2 if l == L - 1 else h) for l in range(L)]
    weights = [((r.standard_normal((27, co, ci)) * math.sqrt(2.0 / (27 * ci))).astype(np.float32),
                (0.01 * r.standard_normal(co)).astype(np.float32)) for ci, co in shapes]
    return x, target, weights


# ------------------------------------------------------------------ prepare and run
def _make_scalar(case):
    m = ONE if case["fields"] == 1 else TWO
    lat = cl.Lattice(case["N"], m["dx"] * case["N"], case["fields"], PREC[case["precision"]],
                     INTEG[case.get("integrator", "vv2")], alpha=m["alpha"], kappa=m["kappa"], dt=m["dt"])
    if case["fields"] == 1:
        lat.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
    else:
        lat.cl_set_potential(cl.CL_POT_M2_G2, [1.0, m["g2"]])
    return lat


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("scalar", "spectra"):
        lat = _make_scalar(case)
        phi, pi = _scalar_inputs(case["N"], case["fields"], case["precision"], seed)
        fields = [(cl.CL_FIELD_PHI0 + f, x) for f, x in enumerate(phi)]
        fields += [(cl.CL_FIELD_PI0 + f, x) for f, x in enumerate(pi)]
        if case.get("gw"):
            lat.cl_enable_gw()
            zero = torch.zeros_like(phi[0])  # no waves at the start
            fields += [(f, zero) for f in range(cl.CL_FIELD_GW_V11, cl.CL_FIELD_GW_P23 + 1)]
        if kind == "spectra":
            for f, x in fields:
                lat.cl_set_state(f, x)
            lat.cl_sync()
    elif kind == "u1":
        N = case["N"]
        lat = cl.Lattice(N, U1["dx"] * N, 1, PREC[case["precision"]], INTEG[case["integrator"]],
                         gauge=cl.CL_GAUGE_U1_AXION, alpha=U1["alpha"], kappa=U1["kappa"], dt=U1["dt"])
        lat.cl_set_potential(cl.CL_POT_M2, [1.0])
        lat.cl_set_gauge_coupling(U1["alphaL"], U1["ws2"])
        phi, pi, theta, E = _u1_inputs(N, case["precision"], seed)
        fields = [(cl.CL_FIELD_PHI0, phi), (cl.CL_FIELD_PI0, pi)]
        fields += [(cl.CL_FIELD_THETA1 + i, x) for i, x in enumerate(theta)]
        fields += [(cl.CL_FIELD_E1 + i, x) for i, x in enumerate(E)]
    elif kind == "ensemble":
        sizes, phi, pi = _ensemble_inputs(case, seed)
        lat = cl.Lattice(sizes[0], ONE["dx"] * 32, 1, cl.CL_PREC_FP32_KAHAN, cl.CL_INT_VV2, alpha=ONE["alpha"],
                         kappa=ONE["kappa"], dt=ONE["dt"], member_N=sizes, member_L=[ONE["dx"] * n for n in sizes])
        lat.cl_set_potential(cl.CL_POT_LPHI4, [1.0])
        V = [n ** 3 for n in sizes]
        out = [torch.empty_like(phi), torch.empty_like(pi)]
        st.update(phi=phi.split(V), pi=pi.split(V), out=out, out_phi=out[0].split(V), out_pi=out[1].split(V))
        fields = []
    else:
        x, target, weights = _surrogate_inputs(case, seed)
        net = cl.Surrogate(case["N"], 3, 2, case["hidden"], case["layers"], ACT[case["activation"]], cl.CL_SG_BF16)
        for l, (W, b) in enumerate(weights):
            net.set_weights(l, W, b)
        st.update(net=net, x=x, target=target, y=torch.empty_like(target))
        return st
    st.update(lat=lat, fields=fields)
    if kind in ("scalar", "u1"):
        st["out"] = [torch.empty_like(x) for _, x in fields]
    return st


ENERGY_KEYS = ("t", "a", "adot", "K0", "K1", "G0", "G1", "V", "KE", "GB", "rho", "p")


def _energy_row(e):
    return [e[k] for k in ENERGY_KEYS]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "surrogate":
        net = state["net"]
        net.forward(state["x"], state["y"])
        loss = net.loss(state["target"])
        net.backward_from_loss()
        return [state["y"], loss] + [net.grads(l) for l in range(case["layers"])]
    lat = state["lat"]
    if kind == "spectra":
        return [lat.cl_spectrum(f) for f, _ in state["fields"]]
    if kind == "ensemble":
        for m in range(case["members"]):
            lat.cl_set_state(cl.CL_FIELD_PHI0, state["phi"][m], member=m)
            lat.cl_set_state(cl.CL_FIELD_PI0, state["pi"][m], member=m)
        lat.cl_set_scalars(1.0, member=-1)
        lat.cl_step(case["steps"])
        for m in range(case["members"]):
            lat.cl_get_state(cl.CL_FIELD_PHI0, state["out_phi"][m], member=m)
            lat.cl_get_state(cl.CL_FIELD_PI0, state["out_pi"][m], member=m)
        return state["out"] + [np.array([_energy_row(e) for e in lat.cl_energies(case["members"])])]
    for f, x in state["fields"]:
        lat.cl_set_state(f, x)
    lat.cl_set_scalars(1.0)
    lat.cl_step(case["steps"])
    for (f, _), y in zip(state["fields"], state["out"]):
        lat.cl_get_state(f, y)
    return state["out"] + [np.array(_energy_row(lat.cl_energies()))]


# ------------------------------------------------------------------ work
def work(case):
    """Bytes: the fields in and out once, and every pass's (stage's) read and write of the state
    (the expansion couples each pass to the volume averages of the one before)."""
    kind = case["kind"]
    if kind == "surrogate":
        V, h = case["N"] ** 3, case["hidden"]
        pairs = 3 * h + (case["layers"] - 2) * h * h + 2 * h
        return {"bytes": V * (4.0 * (3 + 2 + 2) + 2.0 * 2 * 2 * h * (case["layers"] - 1)),
                "flops": 2.0 * 27 * V * (3 * pairs - 3 * h)}  # forward, data and weight gradients
    if kind == "spectra":
        V, es = case["N"] ** 3, 8 if case["precision"] == "fp64" else 4
        return {"bytes": 2.0 * case["fields"] * V * es,
                "flops": 2 * case["fields"] * (2.5 * V * math.log2(V) + 2.0 * V)}
    if kind == "ensemble":
        V = sum(n ** 3 for n in _ensemble_sizes(case))
        return {"bytes": V * (24.0 * case["steps"] + 16.0), "flops": 40.0 * V * case["steps"]}
    V, es = case["N"] ** 3, 8 if case["precision"] == "fp64" else 4
    passes = PASSES[case["integrator"]] * case["steps"]
    if kind == "u1":
        # Runge-Kutta: 8 degrees of freedom and their auxiliaries (the first stage of a step reads
        # none); leapfrog: 16 + 16 + 20 arrays in the three force evaluations of a step
        arrays = 52 * case["steps"] if case["integrator"] == "vv2" else 32 * passes - 8 * case["steps"]
        evals = 3 * case["steps"] if case["integrator"] == "vv2" else passes
        return {"bytes": V * es * (arrays + 16.0), "flops": 500.0 * V * evals}
    nf = case["fields"]
    per = 3 if case["precision"] == "fp32k" else 2
    arrays = 2 * nf * (per + 2) * passes - 2 * nf * case["steps"] if case["integrator"].startswith("rk") else \
        2 * nf * per * passes
    flops = 40.0 * nf * passes
    inout = 4 * nf
    if case["gw"]:
        arrays += (20 + nf) * passes
        flops += 110.0 * passes
        inout += 20
    return {"bytes": float(V * es * (arrays + inout)), "flops": V * flops}


# ------------------------------------------------------------------ the same in 64 bits
def _fwd(f, d):  # f(n + e_d); direction 0 is the fastest index
    return torch.roll(f, -1, 2 - d)


def _back(f, d):
    return torch.roll(f, 1, 2 - d)


def _lap(f, dx):
    s = -6.0 * f
    for d in range(3):
        s += _fwd(f, d)
        s += _back(f, d)
    return s / dx ** 2


def _grad2(f):
    return sum(float((_fwd(f, d) - f).square().sum()) for d in range(3))


class _Exact:
    """The equations of motion in 64 bits: scalars, and the axion-U(1) system where th is given."""

    def __init__(self, model, fields, phi, pi, th=None, E=None, gw=False, dx=None):
        self.m, self.nf, self.phi, self.pi, self.th, self.E = model, fields, phi, pi, th, E
        self.al, self.kappa, self.dx = model["alpha"], model["kappa"], model["dx"] if dx is None else dx
        self.a, self.b, self.t = 1.0, 0.0, 0.0
        self.v = [torch.zeros_like(phi[0]) for _ in range(5)] if gw else None
        self.pv = [torch.zeros_like(phi[0]) for _ in range(5)] if gw else None
        e = self.energies()
        self.b = self.a * self.a ** self.al * math.sqrt(self.kappa * e["rho"] / 3.0)

    def potential(self):
        if self.th is not None:
            return 0.5 * self.phi[0].square()
        if self.nf == 1:
            return 0.25 * self.phi[0].square().square()
        return 0.5 * self.phi[0].square() + 0.5 * self.m["g2"] * (self.phi[0] * self.phi[1]).square()

    def dV(self, f):
        if self.th is not None:
            return self.phi[0]
        if self.nf == 1:
            return self.phi[0] ** 3
        if f == 0:
            return self.phi[0] * (1.0 + self.m["g2"] * self.phi[1].square())
        return self.m["g2"] * self.phi[0].square() * self.phi[1]

    def plaquettes(self, th):
        """theta of the plaquette of normal k at its lower corner."""
        r = []
        for k in range(3):
            i, j = (k + 1) % 3, (k + 2) % 3
            r.append(th[i] + _fwd(th[j], i) - _fwd(th[i], j) - th[j])
        return r

    def energies(self):
        V, a = float(self.phi[0].numel()), self.a
        e = dict.fromkeys(ENERGY_KEYS, 0.0)
        for f in range(self.nf):
            e["K%d" % f] = float(self.pi[f].square().sum()) / (2.0 * a ** 6 * V)
            e["G%d" % f] = _grad2(self.phi[f]) / self.dx ** 2 / (2.0 * a * a * V)
        e["V"] = float(self.potential().sum()) / V
        if self.th is not None:
            w = self.m["ws2"]
            e["KE"] = w * sum(float(x.square().sum()) for x in self.E) / (2.0 * a ** (2 + 2 * self.al) * V)
            e["GB"] = w * sum(float((0.5 * p).sin().square().sum()) for p in self.plaquettes(self.th)) * 2.0 / \
                self.dx ** 4 / (a ** 4 * V)
        K, G, em = e["K0"] + e["K1"], e["G0"] + e["G1"], e["KE"] + e["GB"]
        e["rho"], e["p"] = K + G + e["V"] + em, K - G / 3.0 - e["V"] + em / 3.0
        e["t"], e["a"], e["adot"] = self.t, a, self.b
        return e

    def addot(self):
        e = self.energies()
        return self.a ** (2 * self.al + 1) * self.kappa / 6.0 * ((2 * self.al - 1) * e["rho"] - 3.0 * e["p"])

    def force(self, f):
        return self.a ** (1 + self.al) * _lap(self.phi[f], self.dx) - self.a ** (3 + self.al) * self.dV(f)

    def gw_force(self):
        c = self.a ** (1 + self.al)
        Pi = {}
        for f in range(self.nf):
            d = [(_fwd(self.phi[f], k) - _back(self.phi[f], k)) / (2 * self.dx) for k in range(3)]
            for i in range(3):
                for j in range(i, 3):
                    Pi[i, j] = Pi.get((i, j), 0.0) + d[i] * d[j]
        tr = (Pi[0, 0] + Pi[1, 1] + Pi[2, 2]) / 3.0
        ij = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2))
        return [c * _lap(v, self.dx) + 2.0 * self.kappa * c * (Pi[q] - (tr if q[0] == q[1] else 0.0))
                for v, q in zip(self.v, ij)]

    def kick(self, h):
        F = [self.force(f) for f in range(self.nf)]
        for f in range(self.nf):
            self.pi[f] += h * F[f]
        if self.v:
            for p, x in zip(self.pv, self.gw_force()):
                p += h * x

    def verlet(self, h):
        self.b += 0.5 * h * self.addot()
        self.kick(0.5 * h)
        a1 = self.a + h * self.b
        c = h * (0.5 * (self.a + a1)) ** (self.al - 3.0)
        for f in range(self.nf):
            self.phi[f] += c * self.pi[f]
        for x, p in zip(self.v or (), self.pv or ()):
            x += c * p
        self.a = a1
        self.kick(0.5 * h)
        self.b += 0.5 * h * self.addot()

    def u1_rhs(self, pi, E, b):
        """(pi', E') at the positions of this state, momenta (pi, E) and a' = b."""
        m, dx, a, al, phi = self.m, self.dx, self.a, self.al, self.phi[0]
        g = m["alphaL"] * math.sqrt(self.kappa)
        P, R = self.plaquettes(self.th), self.plaquettes(E)
        s, c = [x.sin() for x in P], [x.cos() for x in P]
        dphi = a ** (al - 3.0) * pi
        dpi = self.force(0)
        mag, cs, W = [0.0] * 3, [0.0] * 3, [0.0] * 3

        def scatter(to, k, x):  # x times the derivative of the plaquette of normal k by its four links
            i, j = (k + 1) % 3, (k + 2) % 3
            to[i] = to[i] + x - _fwd_inv(x, j)
            to[j] = to[j] - x + _fwd_inv(x, i)

        def _fwd_inv(x, d):  # the plaquette at q holds the link at q + e_d
            return _back(x, d)

        for k in range(3):
            i, j = (k + 1) % 3, (k + 2) % 3

            def clover(x):  # the four plaquettes around a site
                y = x + _back(x, i)
                return y + _back(y, j)

            B = clover(s[k]) / (4 * dx * dx)
            Bdot = clover(c[k] * (dx * R[k])) / (4 * dx * dx)
            Eb = 0.5 * (E[k] + _back(E[k], k))
            dpi = dpi + m["ws2"] * g * Eb * B
            scatter(mag, k, s[k] / dx ** 3)
            x = phi * Eb
            x = x + _fwd(x, i)
            x = x + _fwd(x, j)  # the four sites around a plaquette
            scatter(cs, k, x * c[k] / (4 * dx))
            x = dphi * B + phi * Bdot
            W[k] = 0.5 * (x + _fwd(x, k))
        dE = [a ** (al - 1) * (-a ** (al - 1) * mag[k] + g * (cs[k] - W[k])) - (1 - al) * (b / a) * E[k]
              for k in range(3)]
        return dphi, dpi, dE

    def rk(self, A, B, h):
        y = self.phi + self.pi + (self.th + self.E if self.th is not None else [])
        k = [0.0] * len(y)
        ka = kb = 0.0
        for As, Bs in zip(A, B):
            Fa, Fb = self.b, self.addot()
            if self.th is not None:
                dphi, dpi, dE = self.u1_rhs(self.pi[0], self.E, self.b)
                F = [dphi, dpi] + [self.dx * x for x in self.E] + dE
            else:
                F = [self.a ** (self.al - 3.0) * x for x in self.pi] + [self.force(f) for f in range(self.nf)]
            for q in range(len(y)):
                k[q] = As * k[q] + h * F[q]
            for q in range(len(y)):
                y[q] += Bs * k[q]
            ka, kb = As * ka + h * Fa, As * kb + h * Fb
            self.a, self.b = self.a + Bs * ka, self.b + Bs * kb

    def u1_leapfrog(self, h, steps):
        """Implicit half-kick by three evaluations, drift, explicit half-kick."""
        _, gp, gE = self.u1_rhs(self.pi[0], self.E, self.b)
        for _ in range(steps):
            bh = self.b + 0.5 * h * self.addot()
            pk, Ek = self.pi[0] + 0.5 * h * gp, [e + 0.5 * h * x for e, x in zip(self.E, gE)]
            for _ in range(2):
                _, gp, gE = self.u1_rhs(pk, Ek, bh)
                pk, Ek = self.pi[0] + 0.5 * h * gp, [e + 0.5 * h * x for e, x in zip(self.E, gE)]
            a1 = self.a + h * bh
            self.phi[0] = self.phi[0] + h * (0.5 * (self.a + a1)) ** (self.al - 3.0) * pk
            self.th = [t + h * self.dx * x for t, x in zip(self.th, Ek)]
            self.a, self.b = a1, bh
            _, gp, gE = self.u1_rhs(pk, Ek, bh)
            self.pi[0] = pk + 0.5 * h * gp
            self.E = [e + 0.5 * h * x for e, x in zip(Ek, gE)]
            self.b = bh + 0.5 * h * self.addot()

    def advance(self, integrator, steps):
        h = self.m["dt"]
        if integrator == "vv2" and self.th is not None:
            self.u1_leapfrog(h, steps)
        elif integrator.startswith("rk"):
            A, B = RK[integrator]
            for _ in range(steps):
                self.rk(A, B, h)
        else:
            w1 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
            for _ in range(steps):
                for w in ((1.0,) if integrator == "vv2" else (w1, 1.0 - 2.0 * w1, w1)):
                    self.verlet(w * h)
        self.t = steps * h
        return self.energies()


# low-storage coefficients: Williamson (1980), Carpenter and Kennedy (1994)
RK = {"rk3-3": ((0.0, -5.0 / 9.0, -153.0 / 128.0), (1.0 / 3.0, 15.0 / 16.0, 8.0 / 15.0)),
      "rk4-5": ((0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
                 -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0),
                (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0,
                 1720146321549.0 / 2090206949498.0, 3134564353537.0 / 4481467310338.0,
                 2277821191437.0 / 14882151754819.0))}


def _conv(h, W, flip=False):
    """Periodic 3x3x3 convolution of (z, y, x, c) by taps; flip: its adjoint."""
    out = 0.0
    for t in range(27):
        o = (t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1)
        if flip:
            out = out + torch.roll(h, o, (0, 1, 2)) @ W[t]
        else:
            out = out + torch.roll(h, [-x for x in o], (0, 1, 2)) @ W[t].T
    return out


def _exact_surrogate(case, seed):
    x, target, weights = _surrogate_inputs(case, seed)
    x, target = x.double(), target.double()
    w = [(torch.from_numpy(W).to(x.device).double(), torch.from_numpy(b).to(x.device).double()) for W, b in weights]
    L, relu = case["layers"], case["activation"] == "relu"
    c = math.sqrt(2.0 / math.pi)
    acts, pre = [x], []
    for l in range(L - 1):
        u = _conv(acts[-1], w[l][0]) + w[l][1]
        pre.append(u)
        acts.append(u.clamp(min=0) if relu else 0.5 * u * (1 + torch.tanh(c * (u + 0.044715 * u ** 3))))
    y = x[..., :2] + _conv(acts[-1], w[-1][0]) + w[-1][1]
    loss = float((y - target).square().mean())
    g = 2.0 * (y - target) / target.numel()
    grads = [None] * L
    for l in range(L - 1, -1, -1):
        h, g2 = acts[l], g.reshape(-1, g.shape[-1])
        dW = torch.stack([g2.T @ torch.roll(h, [-(t // 9 - 1), -(t // 3 % 3 - 1), -(t % 3 - 1)],
                                            (0, 1, 2)).reshape(-1, h.shape[-1]) for t in range(27)])
        grads[l] = (dW, g2.sum(0))
        if l:
            g = _conv(g, w[l][0], flip=True)
            u = pre[l - 1]
            if relu:
                g = g * (u > 0)
            else:
                th = torch.tanh(c * (u + 0.044715 * u ** 3))
                g = g * (0.5 * (1 + th) + 0.5 * u * (1 - th * th) * c * (1 + 3 * 0.044715 * u * u))
    return [y, loss] + grads


def _exact_spectrum(f, L):
    """Type I spectrum of unit bins: (2 pi / L) l, l S_l / N^6 and the number of modes."""
    N = f.shape[0]
    F = torch.fft.rfftn(f)
    p = F.real.square() + F.imag.square()
    i = torch.arange(N, device=f.device)
    s = torch.where(i <= N // 2, i, i - N)
    n2 = s[:, None, None] ** 2 + s[None, :, None] ** 2 + s[None, None, : N // 2 + 1] ** 2
    w = torch.full((N // 2 + 1,), 2.0, dtype=torch.float64, device=f.device)
    w[0] = 1.0
    if N % 2 == 0:
        w[N // 2] = 1.0
    l = torch.floor(n2.double().sqrt() + 0.5).long()
    nb = int(math.floor(math.sqrt(3.0) * (N // 2) + 0.5)) + 1
    w = w.expand(l.shape)
    S = torch.bincount(l.reshape(-1), (w * p).reshape(-1), minlength=nb)[:nb]
    C = torch.bincount(l.reshape(-1), w.reshape(-1), minlength=nb)[:nb]
    n = torch.arange(nb, dtype=torch.float64, device=f.device)
    return (2.0 * math.pi / L * n).cpu().numpy(), (n * S / float(N) ** 6).cpu().numpy(), C.cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "surrogate":
        return _exact_surrogate(case, seed)
    if kind == "ensemble":
        sizes, phi, pi = _ensemble_inputs(case, seed)
        V = [n ** 3 for n in sizes]
        ends = []
        for n, p, q in zip(sizes, phi.split(V), pi.split(V)):
            x = _Exact(ONE, 1, [p.double().reshape(n, n, n)], [q.double().reshape(n, n, n)])
            ends.append((x, x.advance("vv2", case["steps"])))
        return [torch.cat([x.phi[0].reshape(-1) for x, _ in ends]), torch.cat([x.pi[0].reshape(-1) for x, _ in ends]),
                np.array([_energy_row(e) for _, e in ends])]
    N = case["N"]
    if kind == "u1":
        phi, pi, theta, E = _u1_inputs(N, case["precision"], seed)
        x = _Exact(U1, 1, [phi.double()], [pi.double()], [t.double() for t in theta], [e.double() for e in E])
        e = x.advance(case["integrator"], case["steps"])
        return x.phi + x.pi + x.th + x.E + [np.array(_energy_row(e))]
    phi, pi = _scalar_inputs(N, case["fields"], case["precision"], seed)
    model = ONE if case["fields"] == 1 else TWO
    if kind == "spectra":
        return [_exact_spectrum(f.double(), model["dx"] * N) for f in phi + pi]
    x = _Exact(model, case["fields"], [f.double() for f in phi], [f.double() for f in pi], gw=case["gw"])
    e = x.advance(case["integrator"], case["steps"])
    return x.phi + x.pi + (x.v + x.pv if case["gw"] else []) + [np.array(_energy_row(e))]
