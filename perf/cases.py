"""Workloads of the FLBM library as its users run them, for timing.

A case is a plain dict. `kind` says which entry point it goes through:

  channel      one simulation on the GPU: `Sim.step` and the particle record (`Sim.particle`)
  ensemble     many simulations in batched launches: `Ensemble.step`, every particle record, a few members' populations
  adjoint      the settling velocity of a noise-free run and its gradient (`settling_velocity`, torch autograd)
  host         a run from host memory and back, with the record of every step (`Sim.run_host`)
  observables  the reduced observables of a state (`Sim.observables`)

`exact` computes the same outputs in FP64 with plain torch operations (`Reference`, a dense restatement of the
method; arXiv:1909.01092, Sections 2 and 3), for every case whose dense run takes seconds.
"""
import math

import numpy as np
import torch

from paper_1909_01092_gb300 import binding, workloads

PAPER_FLUID = dict(G=1.5, rho_a0=2.21, rho_b0=0.09)  # the fluid of Section 3's production runs


def listed():
    return [
        # The noise-free validation channel: the smallest system, all launches and latency.
        dict(name="channel 16x16x32", kind="channel", lx=16, ly=16, lz=32, walls="xy", radius=3.0, kT=0.0,
             wetting=0.0, fluid="dilute", tau=1.0, counterforce=False, steps=16, graphs=True),
        # The fluctuating channel whose velocity statistics are collected over 200k steps.
        dict(name="channel 32x32x64 noise", kind="channel", lx=32, ly=32, lz=64, walls="xy", radius=4.0, kT=1e-5,
             wetting=0.5, fluid="dilute", tau=1.0, counterforce=False, steps=16, graphs=True),
        # The noise-free channel of the gradient studies, run forward only.
        dict(name="channel 64x64x128", kind="channel", lx=64, ly=64, lz=128, walls="xy", radius=8.0, kT=0.0,
             wetting=0.3, fluid="dilute", tau=1.0, counterforce=False, steps=16, graphs=True),
        # The throughput channel: populations of 1.3 GB per copy.
        dict(name="channel 128x128x512 noise", kind="channel", lx=128, ly=128, lz=512, walls="xy", radius=12.0,
             kT=1e-5, wetting=0.0, fluid="dilute", tau=1.0, counterforce=False, steps=8, graphs=True),
        # The closed 60x60x900 production channel of Section 3: ragged rows, walls on every axis.
        dict(name="closed 60x60x900 noise", kind="channel", lx=60, ly=60, lz=900, walls="xyz", radius=8.0, kT=1e-5,
             wetting=0.0, fluid="paper", tau=1.0, counterforce=False, steps=8, graphs=True),
        # A periodic mixture without a particle, three relaxation times different from 1, plain launches.
        dict(name="mixture 100x90x110 mrt", kind="channel", lx=100, ly=90, lz=110, walls="", radius=0.0, kT=1e-5,
             wetting=0.0, fluid="paper", tau=0.8, counterforce=False, steps=8, graphs=False),
        # The uneven replicas of the batched ensemble (cross-sections 16 to 48, radii 2.5 to 6), tuned configuration.
        dict(name="ensemble 128 replicas", kind="ensemble", members="uneven", n=128, L=0, lz=0, kT=0.0, packing=0,
             ctas_per_sm=0, tile_policy=1, steps=16),
        # The confinement study's channels (five diameters, three wettings) in one ensemble, default configuration.
        dict(name="ensemble confinement", kind="ensemble", members="confinement", n=15, L=60, lz=120, kT=4.5e-4,
             packing=0, ctas_per_sm=4, tile_policy=0, steps=16),
        # The gradient on a channel small enough for finite differences.
        dict(name="adjoint 16x16x32", kind="adjoint", lx=16, ly=16, lz=32, radius=3.0, wetting=0.3, steps=48,
             checkpoint_every=16),
        # The gradient study's channel, its tape kept whole.
        dict(name="adjoint 64x64x128", kind="adjoint", lx=64, ly=64, lz=128, radius=8.0, wetting=0.3, steps=100,
             checkpoint_every=50),
        # A run from pinned host memory with the trajectory, as a host program calls the C ABI.
        dict(name="host 64x64x128 noise", kind="host", lx=64, ly=64, lz=128, walls="xy", radius=8.0, kT=1e-5,
             wetting=0.0, fluid="dilute", steps=48),
        # Masses, momentum and the temperatures of every mode of a large state.
        dict(name="observables 128x128x128", kind="observables", lx=128, ly=128, lz=128, walls="xy", radius=12.0,
             fluid="dilute"),
    ]


def draw(rng):
    kind = rng.choice(["channel"] * 5 + ["ensemble"] * 2 + ["adjoint"] * 2 + ["host", "observables"])
    if kind == "ensemble":
        policy, ctas = rng.choice([(0, 4), (1, 0), (0, 0), (1, 2)])
        cfg = dict(kind=kind, packing=rng.randrange(3), ctas_per_sm=ctas, tile_policy=policy)
        if rng.random() < 0.5:
            return dict(cfg, members="uneven", n=rng.randrange(4, 129), L=0, lz=0, kT=0.0,
                        steps=2 * rng.randrange(1, 9))
        return dict(cfg, members="confinement", n=15, L=rng.randrange(30, 61), lz=rng.randrange(48, 121),
                    kT=rng.choice([1e-5, 4.5e-4]), steps=2 * rng.randrange(1, 9))
    if kind == "adjoint":
        s = math.exp(rng.uniform(math.log(14), math.log(64)))
        lx, ly = (max(14, round(s * rng.uniform(0.85, 1.1))) for _ in range(2))
        lz = min(128, max(20, round(2 * s * rng.uniform(0.8, 1.1))))
        return dict(kind=kind, lx=lx, ly=ly, lz=lz, radius=round(min(lx, ly) * rng.uniform(0.13, 0.2), 2),
                    wetting=rng.choice([0.0, 0.1, 0.3]), steps=rng.randrange(20, 61),
                    checkpoint_every=rng.randrange(10, 41))
    top = {"channel": 8.0e6, "host": 1.0e6, "observables": 4.0e6}[kind]
    nodes = math.exp(rng.uniform(math.log(5e3), math.log(top)))
    s = nodes ** (1.0 / 3.0)
    lx, ly = (max(12, round(s * rng.uniform(0.45, 1.0))) for _ in range(2))
    lz = max(16, int(nodes / (lx * ly)))
    radius = round(rng.uniform(0.12, 0.25) * min(lx, ly, lz, 60), 2)
    c = dict(kind=kind, lx=lx, ly=ly, lz=lz, walls=rng.choice(["xy", "xy", "xyz", "y", ""]), radius=radius,
             fluid=rng.choice(["dilute", "paper"]))
    if kind == "observables":
        return c
    c.update(kT=rng.choice([0.0, 1e-6, 1e-5, 1e-4]), wetting=rng.choice([0.0, 0.05, 0.3]))
    if kind == "host":
        return dict(c, steps=8 * rng.randrange(1, 7))
    if rng.random() < 0.25:
        c["radius"] = 0.0
    return dict(c, tau=rng.choice([1.0, 1.0, 1.0, 0.8]), counterforce=bool(c["radius"]) and rng.random() < 0.3,
                steps=2 * rng.randrange(1, 9) if nodes < 1e6 else 2 * rng.randrange(1, 4),
                graphs=rng.random() < 0.75)


# ---------------------------------------------------------------------------
# Inputs from a seed
# ---------------------------------------------------------------------------
def start_of(case, seed):
    """Parameters of a channel, and the sphere's position, velocity and spin: it is moving, off the centre."""
    rng = np.random.default_rng(seed)
    walls = case.get("walls", "xy")
    fluid = PAPER_FLUID if case.get("fluid") == "paper" else {}
    tau = case.get("tau", 1.0)
    # tau stands for three different relaxation times once it leaves 1
    taus = dict(tau_s=tau, tau_d=1.0 + (tau - 1.0) / 2, tau_g=1.0 - (tau - 1.0) / 2)
    centre = [(case[k] - 1) / 2.0 for k in ("lx", "ly", "lz")]
    pos0 = [c + rng.uniform(-0.5, 0.5) for c in centre]
    # Driven to a few hundredths of a lattice unit per step, so that nodes are covered and uncovered as it goes;
    # in a closed channel the paper's weak drive, which keeps it away from the end walls.
    ratio = 2.0 if fluid else 1.5
    g = 5e-6 if "z" in walls or not case["radius"] else 0.03 / ((ratio - 1.0) * case["radius"] ** 2)
    p = workloads.params(lx=case["lx"], ly=case["ly"], lz=case["lz"], wall=tuple(int(a in walls) for a in "xyz"),
                         radius=case["radius"], rho_p_ratio=ratio, g=g, kT=case.get("kT", 0.0),
                         delta_rho=case.get("wetting", 0.0), pos0=pos0, seed=seed,
                         fluid_counterforce=int(case.get("counterforce", False)), **taus, **fluid)
    V = (rng.uniform(-8e-3, 8e-3), rng.uniform(-8e-3, 8e-3), rng.uniform(3e-2, 5e-2))
    Om = tuple(rng.uniform(-4e-3, 4e-3, 3))
    return p, V, Om


def members_of(case, seed):
    if case["members"] == "uneven":
        return workloads.ensemble_members(case["n"], seed)
    out = []
    for d_over_L in (0.133, 0.267, 0.4, 0.533, 0.667):
        for wetting in (-0.1, 0.0, 0.1):
            L = case["L"]
            out.append(workloads.params(lx=L, ly=L, lz=case["lz"], radius=0.5 * d_over_L * L, rho_p_ratio=2.0, g=5e-5,
                                        kT=case["kT"], delta_rho=wetting, fluid_counterforce=1, replica=len(out),
                                        seed=seed, **PAPER_FLUID))
    return out


def sampled_members(plist):
    """The members whose populations a pass reads back: the smallest lattice, and the last replica if it is small."""
    nodes = [p["lx"] * p["ly"] * p["lz"] for p in plist]
    return sorted({nodes.index(min(nodes))} | {r for r in (len(plist) - 1,) if nodes[r] <= 100000})


def perturbed(p, seed, device):
    """Populations (float32) of a thermal-like state: every direction within 2 % of its weight, a drift of 1e-2."""
    g = torch.Generator(device=device).manual_seed(seed)
    shape = (p["lz"], p["ly"], p["lx"])
    f = torch.empty((2, 19) + shape, dtype=torch.float32, device=device)
    drift = [0.01 * torch.randn(shape, generator=g, device=device) for _ in range(3)]
    for l, rho in enumerate((p["rho_a0"], p["rho_b0"])):
        for i in range(19):
            v = 1.0 + 3.0 * sum(float(C[i][a]) * drift[a] for a in range(3))
            f[l, i] = W[i] * rho * (v + 0.02 * torch.randn(shape, generator=g, device=device))
    return f


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        cfg = {k: case[k] for k in ("packing", "ctas_per_sm", "tile_policy")}
        plist = members_of(case, seed)
        ens = binding.Ensemble(plist, config=cfg)
        return dict(case=case, ens=ens, read=sampled_members(plist))
    if kind == "adjoint":
        p, V, _ = start_of(case, seed)
        theta = torch.ones(3, dtype=torch.float32, requires_grad=True)
        J = binding.settling_velocity(p, case["steps"], case["checkpoint_every"], v0=V)
        return dict(case=case, J=J, theta=theta, scale=theta_scale(p))
    p, V, Om = start_of(case, seed)
    # Graph replay needs a stream of the caller's; plain launches go to torch's current one.
    stream = torch.cuda.Stream() if case.get("graphs", kind == "host") else torch.cuda.current_stream()
    sim = binding.Sim(p, stream=stream)
    if case["radius"] > 0:
        sim.set_particle(p["pos0"], V, Om)
    if case.get("graphs", kind == "host"):
        sim.use_graphs(True)
    s = dict(case=case, sim=sim)
    if kind == "host":
        s["f_in"] = torch.from_numpy(sim.read_f()).pin_memory().numpy()
        s["f_out"] = torch.empty(sim.shape, dtype=torch.float32, pin_memory=True).numpy()
    elif kind == "observables":
        sim.write_f(perturbed(p, seed, "cuda").cpu().numpy())
    else:
        # The population storage lent to the library holds two copies; after an even number of steps the first is
        # the current one.
        s["f"] = sim._buf.view(torch.float32)[: 38 * sim.N].view(sim.shape)
    return s


def theta_scale(p):
    """What the three design variables of the gradient scale: body force, wetting and coupling (float32 leaves)."""
    return (p["g"], p["delta_rho"], p["G"])


def motion(recs):
    """Centres, rigid-body velocities (V, Omega) and step-averaged velocities of particle records, as float32 arrays."""
    return dict(X=np.array([r["X"] for r in recs], dtype=np.float32),
                velocity=np.array([np.concatenate([r["V"], r["Omega"]]) for r in recs], dtype=np.float32),
                Vavg=np.array([r["Vavg"] for r in recs], dtype=np.float32))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "channel":
        sim = s["sim"]
        sim.step(case["steps"])
        if case["radius"] > 0:
            return dict(motion([sim.particle()]), f=s["f"])
        return dict(f=s["f"])
    if kind == "ensemble":
        s["ens"].step(case["steps"])
        return dict(motion(s["ens"].particles()), f=[s["ens"].read_f(r) for r in s["read"]])
    if kind == "adjoint":
        th = s["theta"]
        th.grad = None
        J = s["J"](*(th[k] * s["scale"][k] for k in range(3)))
        J.backward()
        return dict(J=J.detach().float(), grad=th.grad)
    if kind == "host":
        traj = s["sim"].run_host(s["f_in"], case["steps"], s["f_out"], traj=True)
        return dict(motion(traj), f=s["f_out"])
    o = s["sim"].observables()
    return {k: o[k] for k in OBS}


OBS = ("mass", "momentum", "kinetic", "nfluid", "nonfinite", "mode_temp", "diff_temp", "mom_temp", "n_bulk")


def work(case):
    """Per node and step: 38 populations read and written; the adjoint also writes and reads the eight moments of the
    tape and reads and writes eight adjoint values. About 900 operations per node, 1700 with the noise."""
    kind = case["kind"]
    steps = case.get("steps", 1)
    if kind == "ensemble":
        nodes = sum(p["lx"] * p["ly"] * p["lz"] for p in members_of(case, 0))
        flops = 1700 if case["kT"] > 0 or case["members"] == "uneven" else 900
        return {"bytes": 304.0 * nodes * steps, "flops": float(flops) * nodes * steps}
    nodes = case["lx"] * case["ly"] * case["lz"]
    if kind == "adjoint":
        return {"bytes": (304.0 + 64.0 + 128.0) * nodes * steps, "flops": 2500.0 * nodes * steps}
    if kind == "observables":
        return {"bytes": 152.0 * nodes, "flops": 400.0 * nodes}
    flops = 1700.0 if case["kT"] > 0 else 900.0
    host = 304.0 * nodes if kind == "host" else 0.0
    return {"bytes": 304.0 * nodes * steps + host, "flops": flops * nodes * steps}


# ---------------------------------------------------------------------------
# The method in FP64
# ---------------------------------------------------------------------------
C = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1))
OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def basis():
    """Rows e_k(c_i) of the D3Q19 mode basis."""
    c = np.array(C, dtype=np.float64)
    x, y, z = c.T
    q = (c * c).sum(1)
    d, e = 3 * x * x - q, y * y - z * z
    rows = [np.ones(19), x, y, z, q - 1, d, e, x * y, y * z, x * z, (3 * q - 5) * x, (3 * q - 5) * y, (3 * q - 5) * z,
            (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z, 3 * q * q - 6 * q + 1, (2 * q - 3) * d,
            (2 * q - 3) * e]
    return np.array(rows)


def philox(ctr, key):
    """Philox4x32-10 on int64 tensors (or ints) holding 32-bit words."""
    m = 0xFFFFFFFF
    x0, x1, x2, x3 = ctr
    k0, k1 = key

    def product(a, v):  # high and low words of the 64-bit product, by 16-bit halves
        a0, a1 = a & 0xFFFF, a >> 16
        p0, p1 = a0 * v, a1 * v
        mid = (p0 >> 16) + (p1 & 0xFFFF)  # p0 < 2^48, p1 < 2^48
        return ((p1 >> 16) + (mid >> 16)) & m, (p0 + ((p1 & 0xFFFF) << 16)) & m

    for _ in range(10):
        h0, l0 = product(0xD2511F53, x0)
        h1, l1 = product(0xCD9E8D57, x2)
        x0, x1, x2, x3 = h1 ^ x1 ^ k0, l1, h0 ^ x3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return x0, x1, x2, x3


def uniform(x):
    return ((x >> 9).double() + 0.5) * 2.0 ** -23


class Reference:
    """One simulation in FP64, dense tensors of (z, y, x). The parameters g, delta_rho and G may be tensors that
    require a gradient: the step is differentiable, with its sets of particle nodes held fixed."""

    def __init__(self, p, device, g=None, delta_rho=None, G=None):
        self.p, self.dev = p, device
        f64 = dict(dtype=torch.float64, device=device)
        as64 = lambda v: v if isinstance(v, torch.Tensor) else torch.tensor(float(v), **f64)  # noqa: E731
        self.g, self.G = as64(p["g"] if g is None else g), as64(p["G"] if G is None else G)
        self.drho = as64(p["delta_rho"] if delta_rho is None else delta_rho)
        self.L = (p["lx"], p["ly"], p["lz"])
        lx, ly, lz = self.L
        self.N = lx * ly * lz
        z, y, x = torch.meshgrid(*(torch.arange(n, device=device) for n in (lz, ly, lx)), indexing="ij")
        self.pos = (x.double(), y.double(), z.double())
        self.node = x + lx * (y + ly * z)
        self.key = (p["seed"] & 0xFFFFFFFF, ((p["seed"] >> 32) ^ p["replica"]) & 0xFFFFFFFF)
        self.wall = p["wall"]
        self.step_no = 0
        # the initial populations are float32 values
        r = philox((0, self.node, 0, 1), self.key)
        self.f = torch.empty((2, 19, lz, ly, lx), **f64)
        for l, rho in enumerate((p["rho_a0"], p["rho_b0"])):
            v = (1.0 + float(np.float32(p["init_pert"])) * (2.0 * uniform(r[l]) - 1.0)).float()
            v = v * float(np.float32(rho))
            for i in range(19):
                self.f[l, i] = (v * float(np.float32(W[i]))).double()
        self.older = self.f  # the other copy: particle nodes keep what it holds
        self.R = p["radius"]
        self.E = torch.tensor(basis(), **f64)
        self.b = (self.E ** 2 * torch.tensor(W, **f64)).sum(1)
        self.delta = torch.zeros(2, **f64)
        self.has = self.R > 0
        self.rho0 = (p["rho_a0"], p["rho_b0"])
        zero = torch.zeros(3, **f64)
        self.X = torch.tensor(p["pos0"], **f64)
        self.V, self.Om, self.Ppend, self.Lpend, self.Vavg = zero, zero, zero, zero, zero
        self.solid = torch.zeros((lz, ly, lx), dtype=torch.bool, device=device)
        if self.has:
            rt0 = sum(self.rho0)
            vol = 4.0 / 3.0 * math.pi * self.R ** 3
            self.mp = vol * p["rho_p_ratio"] * rt0
            self.Ip = 0.4 * self.mp * self.R ** 2
            self.Fp = vol * (p["rho_p_ratio"] - 1.0) * rt0 * self.g
            self.solid = self.inside()
        self.fc = self.counterforce()

    def counterforce(self):
        if not (self.has and self.p["fluid_counterforce"]):
            return 0.0
        return -self.Fp / float(self.N - int(self.solid.sum()))

    def set_particle(self, X, V, Om=(0.0, 0.0, 0.0)):
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=self.dev)  # noqa: E731
        self.X, self.V, self.Om = t(X), t(V), t(Om)
        self.solid = self.inside()
        self.fc = self.counterforce()

    def rel(self, X):
        """Node minus X on each axis, the nearest image on periodic axes."""
        out = []
        for a in range(3):
            d = self.pos[a] - X[a]
            if not self.wall[a]:
                h, L = 0.5 * self.L[a], self.L[a]
                d = torch.where(d > h, d - L, torch.where(d < -h, d + L, d))
            out.append(d)
        return out

    def inside(self):
        with torch.no_grad():
            r = self.rel(self.X)
            return r[0] ** 2 + r[1] ** 2 + r[2] ** 2 < self.R ** 2

    def pad(self, t):
        """One node more on every side of the last three axes: wrapped on periodic axes, zero beyond walls."""
        for a in range(3):
            d = t.dim() - 1 - a
            lo, hi = t.narrow(d, t.shape[d] - 1, 1), t.narrow(d, 0, 1)
            if self.wall[a]:
                lo, hi = torch.zeros_like(lo), torch.zeros_like(hi)
            t = torch.cat([lo, t, hi], d)
        return t

    def at(self, padded, i, sign=1):
        """The interior's neighbours x + sign c_i out of a padded tensor."""
        for a in range(3):
            d = padded.dim() - 1 - a
            padded = padded.narrow(d, 1 + sign * C[i][a], padded.shape[d] - 2)
        return padded

    def densities(self, rho, fluid):
        """The padded density field of the Shan-Chen force: virtual layer on particle nodes, neutral wall ghosts."""
        # two layers around, so that the mean over the neighbours exists on the first
        m = fluid.double()
        S, Cn = self.pad2(rho * m), self.pad2(m)
        s = sum(self.at(S, i) for i in range(1, 19))
        n = sum(self.at(Cn, i) for i in range(1, 19))
        mean = torch.where(n > 0, s / n.clamp(min=1.0), torch.zeros_like(s))
        inside = self.pad(torch.ones_like(m)) > 0  # wrapped copies count as inside
        fl = self.pad(m) > 0
        shift = torch.stack([self.drho, -self.drho]).view(2, 1, 1, 1)
        virt = torch.where(n > 0, (mean + shift).clamp(min=0.0), torch.zeros_like(mean))
        return torch.where(fl, self.pad(rho), torch.where(inside, virt, mean))

    def pad2(self, t):
        """Two nodes more on every side, as `pad`."""
        for a in range(3):
            d = t.dim() - 1 - a
            k = t.shape[d]
            if self.wall[a]:
                z = torch.zeros_like(t.narrow(d, 0, 1))
                t = torch.cat([z, z, t, z, z], d)
            else:
                idx = torch.arange(-2, k + 2, device=self.dev) % k
                t = t.index_select(d, idx)
        return t

    def normals(self):
        """The 33 normals of every node in their order: modes 4..18 of A, of B, interdiffusion."""
        z = []
        for blk in range(9):
            r = philox((self.step_no & 0xFFFFFFFF, self.node, blk, 0), self.key)
            for q in (0, 2):
                rad = torch.sqrt(-2.0 * torch.log(uniform(r[q])))
                ang = 2.0 * math.pi * uniform(r[q + 1])
                z += [rad * torch.cos(ang), rad * torch.sin(ang)]
        return z

    def step(self):
        p = self.p
        fluid = ~self.solid
        rho = self.f.sum(1)
        psi = self.densities(torch.where(fluid, rho, torch.zeros_like(rho)), fluid)
        m = torch.einsum("ki,lizyx->lkzyx", self.E, self.f)
        zero = torch.zeros_like(m[0, 0])
        rl = torch.where(fluid, m[:, 0], torch.ones_like(rho))  # particle nodes are masked out below
        rt = rl[0] + rl[1]
        nb = {i: self.at(psi, i) for i in range(1, 19)}
        grad = [sum(C[i][a] * W[i] * nb[i] for i in range(1, 19) if C[i][a]) for a in range(3)]
        F = []
        for a in range(3):
            ext = p["fluid_force"][a] + (self.fc if a == 2 else 0.0)
            F.append(-self.G * rl * grad[a].flip(0) + rl / rt * ext)
        u = [(m[0, 1 + a] + m[1, 1 + a] + 0.5 * (F[a][0] + F[a][1])) / rt for a in range(3)]
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        gs, gd, gg = (1.0 - 1.0 / p[k] for k in ("tau_s", "tau_d", "tau_g"))
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        eq = [uu, 3 * u[0] ** 2 - uu, u[1] ** 2 - u[2] ** 2, u[0] * u[1], u[1] * u[2], u[0] * u[2]]
        S = [2 * uF, 2 * (3 * u[0] * F[0] - uF), 2 * (u[1] * F[1] - u[2] * F[2]), u[0] * F[1] + u[1] * F[0],
             u[1] * F[2] + u[2] * F[1], u[0] * F[2] + u[2] * F[0]]
        n = [rl + self.delta.view(2, 1, 1, 1)]
        for a in range(3):
            n.append(rl * u[a] + gd * (m[:, 1 + a] + 0.5 * F[a] - rl * u[a]) + 0.5 * F[a])
        for k in range(6):
            n.append(rl * eq[k] + gs * (m[:, 4 + k] - rl * eq[k]) + 0.5 * (1.0 + gs) * S[k])
        for k in range(10, 19):
            n.append(gg * m[:, k])
        n = [v / self.b[k] for k, v in enumerate(n)]
        if p["kT"] > 0:
            z = self.normals()
            amp = torch.sqrt(3.0 * p["kT"] * rl.clamp(min=0.0))
            for k in range(4, 19):
                gk = gs if k <= 9 else gg
                n[k] = n[k] + amp * math.sqrt((1.0 - gk * gk) / float(self.b[k])) * torch.stack(
                    [z[k - 4], z[15 + k - 4]])
            aj = 3.0 * math.sqrt(1.0 - gd * gd) * torch.sqrt(p["kT"] * rl[0].clamp(min=0) * rl[1].clamp(min=0) / rt)
            for a in range(3):
                n[1 + a] = n[1 + a] + torch.stack([aj * z[30 + a], -aj * z[30 + a]])
        fo = torch.einsum("ik,lkzyx->lizyx", self.E.t() * torch.tensor(W, dtype=torch.float64,
                                                                      device=self.dev)[:, None], torch.stack(n, 1))
        # Streaming, bounce-back and the particle links
        solid_p = self.pad(self.solid.double()) > 0
        lattice_p = self.pad(torch.ones_like(zero)) > 0
        fluid_p = lattice_p & ~solid_p
        r = self.rel(self.X)
        force = torch.zeros(3, dtype=torch.float64, device=self.dev)
        torque = torch.zeros_like(force)
        lost = torch.zeros(2, dtype=torch.float64, device=self.dev)
        back = {}
        for i in range(1, 19):
            wallb = fluid & ~self.at(lattice_p, i)
            link = fluid & self.at(solid_p, i)
            b = fo[:, i]
            if self.has:
                mid = [r[a] + 0.5 * C[i][a] for a in range(3)]
                ub = [self.V[0] + self.Om[1] * mid[2] - self.Om[2] * mid[1],
                      self.V[1] + self.Om[2] * mid[0] - self.Om[0] * mid[2],
                      self.V[2] + self.Om[0] * mid[1] - self.Om[1] * mid[0]]
                corr = 6.0 * W[i] * rl * sum(C[i][a] * ub[a] for a in range(3))
                mag = (2.0 * fo[:, i] - corr).sum(0) + self.G * W[i] * (rl[0] * nb[i][1] + rl[1] * nb[i][0])
                mag = torch.where(link, mag, zero)
                fr = [mag * C[i][a] for a in range(3)]
                force = force + torch.stack([t.sum() for t in fr])
                torque = torque + torch.stack([(mid[1] * fr[2] - mid[2] * fr[1]).sum(),
                                               (mid[2] * fr[0] - mid[0] * fr[2]).sum(),
                                               (mid[0] * fr[1] - mid[1] * fr[0]).sum()])
                lost = lost + torch.where(link, corr, torch.zeros_like(corr)).sum((1, 2, 3))
                b = torch.where(link, fo[:, i] - corr, b)
            back[OPP[i]] = (wallb | link, b)
        new = []
        for i in range(19):
            if i == 0:
                v = fo[:, 0]
            else:
                v = self.at(self.pad(fo[:, i]), i, -1)
                came = self.at(fluid_p, i, -1)
                at_wall, b = back[i]
                v = torch.where(at_wall, b, torch.where(came, v, self.older[:, i]))
            new.append(torch.where(fluid, v, self.older[:, i]))
        new = torch.stack(new, 1)
        self.older, self.f = self.f, new
        self.step_no += 1
        if self.has:
            self.advance(force, torque, lost)

    def advance(self, force, torque, lost):
        F, T = force + self.Ppend, torque + self.Lpend
        drive = torch.stack([torch.zeros_like(self.Fp), torch.zeros_like(self.Fp), self.Fp])
        V = self.V + (F + drive) / self.mp
        self.Vavg, self.V = 0.5 * (self.V + V), V
        self.Om = self.Om + T / self.Ip
        X = self.X + V
        wrap = [0.0 if self.wall[a] else self.L[a] * math.floor(float(X[a].detach()) / self.L[a]) for a in range(3)]
        self.X = X - torch.tensor(wrap, dtype=torch.float64, device=self.dev)
        old, new = self.solid, self.inside()
        r = self.rel(self.X)
        imp, ang = torch.zeros_like(force), torch.zeros_like(force)
        ledger = lost
        covered = new & ~old
        uncovered = old & ~new
        for node in covered.nonzero():
            q = tuple(int(t) for t in node)
            f = self.f[(slice(None), slice(None)) + q]
            j = torch.stack([sum(C[i][a] * f[:, i].sum() for i in range(1, 19) if C[i][a]) for a in range(3)])
            rr = torch.stack([r[a][q] for a in range(3)])
            imp, ang = imp + j, ang + torch.linalg.cross(rr, j)
            ledger = ledger + f.sum(1)
        if bool(uncovered.any()):
            ok = (~new & ~old).double()
            s = self.f.sum(1) * ok
            s, n = self.pad(s), self.pad(ok)
            fills = []
            for node in uncovered.nonzero():
                q = tuple(int(t) for t in node)
                around = [tuple(q[2 - a] + 1 + C[i][a] for a in (2, 1, 0)) for i in range(1, 19)]
                cnt = float(sum(n[t] for t in around))
                rl = (sum(s[(slice(None),) + t] for t in around) / cnt if cnt
                      else torch.tensor(self.rho0, dtype=torch.float64, device=self.dev))
                rr = torch.stack([r[a][q] for a in range(3)])
                ub = self.V + torch.linalg.cross(self.Om, rr)
                c = torch.tensor(C, dtype=torch.float64, device=self.dev)
                cu = c @ ub
                prof = torch.tensor(W, dtype=torch.float64, device=self.dev) * (
                    1.0 + 3.0 * cu + 4.5 * cu ** 2 - 1.5 * (ub @ ub))
                fills.append((q, rl[:, None] * prof[None, :]))
                j = rl.sum() * ub
                imp, ang = imp - j, ang - torch.linalg.cross(rr, j)
                ledger = ledger - rl
            z, y, x = (torch.tensor([q[a] for q, _ in fills], device=self.dev) for a in range(3))
            self.f = self.f.index_put((torch.arange(2, device=self.dev)[:, None, None],
                                       torch.arange(19, device=self.dev)[None, :, None], z, y, x),
                                      torch.stack([v for _, v in fills], 2))
        self.solid = new
        nf = float(self.N - int(new.sum()))
        self.Ppend, self.Lpend, self.delta = imp, ang, ledger / nf
        self.fc = self.counterforce()

    def motion(self):
        return {k: v.detach().cpu().numpy() for k, v in (("X", self.X), ("V", self.V), ("Vavg", self.Vavg),
                                                         ("Omega", self.Om))}


def exact_observables(p, f, solid, device):
    """The reductions of `Sim.observables` over populations f in FP64."""
    f = f.to(device).double()
    ref = Reference.__new__(Reference)
    ref.wall, ref.dev = p["wall"], device
    fluid = ~solid
    near = sum(ref.at(ref.pad(solid.double()), i) for i in range(1, 19)) > 0
    bulk = fluid & ~near
    E = torch.tensor(basis(), dtype=torch.float64, device=device)
    b = (E ** 2 * torch.tensor(W, dtype=torch.float64, device=device)).sum(1)
    m = torch.einsum("ki,lizyx->lkzyx", E, f)
    rho, j = m[:, 0], m[0, 1:4] + m[1, 1:4]
    rt = rho.sum(0)
    on = lambda t, mask: t[..., mask].sum(-1)  # noqa: E731
    u = j / rt
    uu = (u * u).sum(0)
    eq = [uu, 3 * u[0] ** 2 - uu, u[1] ** 2 - u[2] ** 2, u[0] * u[1], u[1] * u[2], u[0] * u[2]]
    mt = np.zeros((2, 19))
    mass = on(rho, bulk)
    for l in range(2):
        for k in range(4, 19):
            d = m[l, k] - rho[l] * eq[k - 4] if k <= 9 else m[l, k]
            mt[l, k] = float(on(d * d, bulk) / (3.0 * b[k] * mass[l]))
    d = (rho[1] * m[0, 1:4] - rho[0] * m[1, 1:4]) / rt
    host = lambda t: t.cpu().numpy()  # noqa: E731
    return dict(mass=host(on(rho, fluid)), momentum=host(on(j, fluid)),
                kinetic=float(on((j * j).sum(0) / (2.0 * rt), fluid)), nfluid=int(fluid.sum()), nonfinite=0,
                mode_temp=mt, diff_temp=host(on(d * d, bulk) / on(rho[0] * rho[1] / rt, bulk)),
                mom_temp=host(on(j * j, bulk) / on(rt, bulk)), n_bulk=int(bulk.sum()))


#: Node updates (nodes x steps) that the dense FP64 step is run for: a few seconds.
AFFORDABLE = {"channel": 8.0e7, "host": 8.0e7, "adjoint": 6.0e5, "ensemble": 8.0e6}


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    steps = case.get("steps", 1)
    if kind == "ensemble":
        # Of the records and members, the smallest member's populations.
        plist = members_of(case, seed)
        read = sampled_members(plist)
        nodes = [p["lx"] * p["ly"] * p["lz"] for p in plist]
        small = nodes.index(min(nodes))
        ref = Reference(plist[small], device)
        for _ in range(steps):
            ref.step()
        return dict(X=None, velocity=None, Vavg=None,
                    f=[ref.f.cpu().numpy() if r == small else None for r in read])
    p, V, Om = start_of(case, seed)
    if kind == "observables":
        ref = Reference(p, device)
        ref.set_particle(p["pos0"], V, Om)
        return exact_observables(p, perturbed(p, seed, device), ref.solid, device)
    if case["lx"] * case["ly"] * case["lz"] * steps > AFFORDABLE[kind]:
        return None
    if kind == "adjoint":
        theta = torch.ones(3, dtype=torch.float64, requires_grad=True)
        leaf = [(theta[k] * float(np.float32(s))).to(device) for k, s in enumerate(theta_scale(p))]
        ref = Reference(p, device, *leaf)
        ref.set_particle(p["pos0"], V)
        J = 0.0
        for _ in range(steps):
            ref.step()
            J = J + ref.Vavg[2] / steps
        J.backward()
        return dict(J=J.detach().cpu(), grad=theta.grad)
    with torch.no_grad():
        ref = Reference(p, device)
        if ref.has:
            ref.set_particle(p["pos0"], V, Om)
        rec = []
        for _ in range(steps):
            ref.step()
            rec.append(ref.motion())
        out = {}
        if ref.has:
            rec = rec if kind == "host" else rec[-1:]
            out = dict(X=np.array([r["X"] for r in rec]), Vavg=np.array([r["Vavg"] for r in rec]),
                       velocity=np.array([np.concatenate([r["V"], r["Omega"]]) for r in rec]))
        return dict(out, f=ref.f.cpu())
