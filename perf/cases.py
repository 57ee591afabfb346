"""Cases for timing the library the way its users call it.

A case is one of five kinds of work:

* ``steps``   a running simulation advances and its state is read back (a checkpoint);
* ``sweep``   a batch of droplets of different sizes advances together, every member's state is read back;
* ``check``   the convergence check of a batch: pressure jumps and velocity change of every member;
* ``tension`` the measurement of one droplet: profile, bulk pressures, surface of tension;
* ``fields``  the densities and the velocity of a simulation, with its run diagnostics;
* ``host``    the whole method from host buffers to host results.

Simulations go on from pass to pass, as a user's program runs them: a pass of ``steps`` continues where the
last one ended, and the analysis kinds advance by two time steps first, so that every pass measures a new state.

``exact`` is the method itself in plain FP64 torch (periodic shifts of whole arrays).
"""
from __future__ import annotations

import itertools
import math

import torch

from paper_2112_02574_gb300 import binding as B

DEV = "cuda"
STORAGE = {"f32": B.SC_STORE_F32, "f16": B.SC_STORE_F16, "bf16": B.SC_STORE_BF16, "f64": B.SC_STORE_F64}
ELEM = {"f32": 4, "f16": 2, "bf16": 2, "f64": 8}
DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "f64": torch.float64}
PAPER_SIDES = (25, 31, 37, 41, 51, 57, 65)


def listed():
    return [
        # the two-dimensional droplet in FP64: the smallest lattice in use, latency and FP64 arithmetic
        _steps("d2q9_64_f64", 64, 64, 1, "f64", 64, lattice="d2q9", R=12.0, coupling="d2q9"),
        # the benchmark's droplet, FP32 storage: the ordinary run
        _steps("cube128_f32", 128, 128, 128, "f32", 64, R=24.0),
        # the flat interface with the extended forcing stencil and a self coupling, fewer columns than SMs
        _steps("slab64x256_e6_f32", 64, 64, 256, "f32", 64, stencil="e6", coupling="asym", shape="slab"),
        # the largest droplet, FP16 storage, asymmetric couplings
        _steps("cube512_f16", 512, 512, 512, "f16", 16, R=96.0, coupling="asym"),
        # one droplet of the paper's odd sizes (R = L / 4) on its couplings: a lone small simulation
        _steps("cube51_f32", 51, 51, 51, "f32", 64, R=12.75, coupling="paper"),
        # FP64 storage in three dimensions: the reference every reduced-precision result is compared with
        _steps("cube64_f64", 64, 64, 64, "f64", 16, R=16.0, coupling="asym"),
        # the radius sweep: 16 droplets, R = 8 .. 40, cubes of side 4 ceil(R), half of them asymmetric
        {"name": "sweep16_f32", "kind": "sweep", "set": "radii", "members": 16, "rmin": 8.0, "rmax": 40.0,
         "storage": "f32", "nsteps": 32},
        # the paper's sizes 25 .. 65, A-rich and B-rich, one value of the asymmetry
        {"name": "paper_sweep14_f32", "kind": "sweep", "set": "paper", "members": 14, "storage": "f32",
         "nsteps": 32},
        # section 4's convergence check of that sweep, done every 2048 steps: many small calls
        {"name": "paper_check14_f32", "kind": "check", "set": "paper", "members": 14, "storage": "f32"},
        # the measurement at the end of a benchmark step: radial profile and surface of tension at 128^3
        {**_steps("tension128_f32", 128, 128, 128, "f32", 2, R=24.0), "kind": "tension"},
        # density and velocity fields with the run diagnostics at 128^3, 16-bit storage
        {**_steps("fields128_bf16", 128, 128, 128, "bf16", 2, R=24.0, coupling="asym"), "kind": "fields"},
        # the whole method from host memory to host memory on a small droplet
        {**_steps("host64_f32", 64, 64, 64, "f32", 256, R=16.0), "kind": "host"},
    ]


def _steps(name, nx, ny, nz, storage, nsteps, *, lattice="d3q19", stencil="e4", coupling="sym", shape="droplet",
           R=0.0, tau=1.0):
    c = {"kind": "steps", "nx": nx, "ny": ny, "nz": nz, "storage": storage, "nsteps": nsteps, "lattice": lattice,
         "stencil": stencil, "coupling": coupling, "shape": shape, "R": R, "tau": tau}
    return {"name": name, **c} if name else c


def draw(rng):
    """A case of the same ranges: sides over their logarithm, odd and ragged ones, every storage and stencil."""
    def side(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))

    kind = rng.choice(["steps"] * 6 + ["sweep", "sweep", "check", "tension", "tension", "fields", "host"])
    if kind in ("sweep", "check"):
        storage = rng.choice(["f32", "f32", "f16", "bf16"])
        if rng.random() < 0.5:
            return {"kind": kind, "set": "paper", "members": rng.randint(3, 14), "storage": storage, "nsteps": 32,
                    "seed_size": rng.randrange(1000)}
        rmin = rng.uniform(6.0, 14.0)
        return {"kind": kind, "set": "radii", "members": rng.randint(2, 12), "rmin": rmin,
                "rmax": rng.uniform(rmin + 2.0, 36.0), "storage": storage, "nsteps": 32}
    if kind == "steps" and rng.random() < 0.2:  # two dimensions
        n = side(48, 512)
        return _steps("", n, side(48, 512), 1, rng.choice(["f64", "f32"]), 64, lattice="d2q9", R=n / 5.0,
                      coupling="d2q9")
    storage = rng.choice(["f32", "f32", "f32", "f16", "bf16", "f64"] if kind == "steps" else ["f32", "f32", "bf16"])
    cap = {"f64": 96, "host": 96, "tension": 160, "fields": 160}.get("f64" if storage == "f64" else kind, 288)
    # a cube, a cube that the paper's odd sizes stand for, or a ragged box
    form = rng.choice(["cube", "odd", "box", "slab"]) if kind != "host" else rng.choice(["cube", "odd"])
    nx = ny = nz = side(24, cap)
    if form == "cube":
        nx = ny = nz = nx // 4 * 4
    elif form == "odd":
        nx = ny = nz = nx | 1
    else:
        ny, nz = side(24, cap), side(24, cap)
    tau = rng.choice([1.0, 1.0, 1.0, 1.0, 0.9]) if kind == "steps" else 1.0
    c = _steps("", nx, ny, nz, storage, 32 if kind == "steps" else (rng.choice([64, 128, 192]) if kind == "host" else 2),
               stencil=rng.choice(["e4", "e4", "e6"]) if kind == "steps" else "e4",
               coupling=rng.choice(["sym", "asym", "paper"]), shape="slab" if form == "slab" else "droplet",
               R=min(nx, ny, nz) / 4.0, tau=tau)
    return {**c, "kind": kind}


# ------------------------------------------------------------------ the model's parameters
def _couplings(name):
    """G, (G_AA, G_BB), pseudopotential, total density of the runs the library is used for."""
    if name == "sym":
        return 3.6, (0.0, 0.0), B.SC_PSI_EXP, 1.0
    if name == "asym":  # G_AA c_s^2 = -0.2
        return 3.6, (-0.6, 0.0), B.SC_PSI_EXP, 1.0
    if name == "d2q9":
        return 4.2, (0.0, 0.0), B.SC_PSI_N, 1.0
    g = -math.e ** 2  # the paper's couplings at dG_AB = 0.48
    return 1.5, (g * (1.0 - 0.4 * 1.48), g * 0.6), B.SC_PSI_EXP, 2.0


def _members(case):
    """The lattices of a case, as (nx, ny, nz, coupling, shape, R, A-rich)."""
    if "set" not in case:
        return [(case["nx"], case["ny"], case["nz"], case["coupling"], case["shape"], case["R"], True)]
    n, out = case["members"], []
    for k in range(n):
        if case["set"] == "paper":
            j = k + case.get("seed_size", 0)
            L = PAPER_SIDES[(j // 2) % 7]
            out.append((L, L, L, "paper", "droplet", L / 4.0, j % 2 == 0))
        else:
            R = case["rmin"] + (case["rmax"] - case["rmin"]) * k / max(1, n - 1)
            L = 4 * math.ceil(R)
            out.append((L, L, L, "sym" if k % 2 == 0 else "asym", "droplet", R, True))
    return out


def _params(case, m):
    G, G_self, psi, _ = _couplings(m[3])
    tau = case.get("tau", 1.0)
    return B.make_params(m[:3], lattice=B.SC_D2Q9 if case.get("lattice") == "d2q9" else B.SC_D3Q19,
                         stencil=B.SC_FORCE_E6 if case.get("stencil") == "e6" else B.SC_FORCE_E4, psi_self=psi,
                         storage=STORAGE[case["storage"]], tau=(tau, tau), G=G, G_self=G_self)


def _densities(m, seed):
    """Initial densities [nz, ny, nx]: a tanh droplet at the centre node, or a band along z, with noise of 1e-3."""
    nx, ny, nz, coupling, shape, R, a_rich = m
    total = _couplings(coupling)[3]
    ax = [torch.arange(n, dtype=torch.float64, device=DEV) - n // 2 for n in (nz, ny, nx)]
    if shape == "slab":
        d = ax[0].abs()[:, None, None].expand(nz, ny, nx) - nz / 4.0
    else:
        r2 = 0.0
        for k, (a, n) in enumerate(zip(ax, (nz, ny, nx))):
            a = a - n * torch.floor(a / n + 0.5)
            r2 = r2 + (a * a).reshape([-1 if j == k else 1 for j in range(3)])
        d = torch.sqrt(r2) - R
    rich = total * (0.5 - 0.45 * torch.tanh(d))
    poor = total - rich
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    out = []
    for n in ((rich, poor) if a_rich else (poor, rich)):
        out.append(n + 1e-3 * (2.0 * torch.rand((nz, ny, nx), generator=g, dtype=torch.float64, device=DEV) - 1.0))
    return out


# ------------------------------------------------------------------ what a pass does
def prepare(case, seed):
    ms = _members(case)
    ps = [_params(case, m) for m in ms]
    fields = [_densities(m, seed * 1009 + 31 * k) for k, m in enumerate(ms)]
    s = {"case": case, "members": ms}
    if case["kind"] == "host":
        p = ps[0]
        s.update(params=p, nA0=fields[0][0].reshape(-1).cpu().pin_memory(), nB0=fields[0][1].reshape(-1).cpu().pin_memory(),
                 workspace=torch.empty(B.sc_workspace_bytes(p), dtype=torch.uint8, device=DEV),
                 nA=torch.empty(fields[0][0].numel(), dtype=torch.float64).pin_memory(),
                 nB=torch.empty(fields[0][0].numel(), dtype=torch.float64).pin_memory(),
                 result=torch.empty(8, dtype=torch.float64).pin_memory())
        return s
    if "set" in case:
        s["batch"] = B.Batch(ps, fields, device=DEV)
        if case["kind"] == "check":
            s["u"] = [m.moments()[2].clone() for m in s["batch"].members]
        return s
    s["sim"] = B.Simulation(ps[0], *fields[0], device=DEV)
    if case["kind"] == "fields":
        s["u"] = s["sim"].moments()[2].clone()
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "steps":
        state["sim"].step(case["nsteps"])
        return _checkpoint(state["sim"], case)
    if kind == "sweep":
        state["batch"].step(case["nsteps"])
        return [_checkpoint(m, case) for m in state["batch"].members]
    if kind == "check":
        batch = state["batch"]
        batch.step(2)
        dp, du = [], []
        for m, u, (nx, ny, nz, *_) in zip(batch.members, state["u"], state["members"]):
            dp.append(m.bulk_pressure((nx // 2, ny // 2, nz // 2)) - m.bulk_pressure((nx - 1, ny - 1, nz - 1)))
            du.append(m.velocity_change(u))
        return {"dP": torch.cat(dp), "dU": torch.cat(du), "u": state["u"]}
    if kind == "tension":
        sim = state["sim"]
        sim.step(case["nsteps"])
        if case["shape"] == "slab":
            rows, out = B.sigma0_flat(sim)
        else:
            rows, out = B.surface_of_tension(sim)
        return {"rows": rows, "result": out}
    if kind == "fields":
        sim = state["sim"]
        sim.step(case["nsteps"])
        nA, nB, u = sim.moments()
        out = torch.empty(10, dtype=torch.float64, device=DEV)
        B.sc_diagnostics(sim.ctx, state["u"], 0, 0.05, out)
        return {"nA": nA, "nB": nB, "u": u, "mass": out[:2], "momentum": out[2:5], "dU": out[5:6], "centre": out[6:]}
    B.sc_run_host_sigma(state["params"], state["nA0"], state["nB0"], case["nsteps"], None, 0.5, 0, state["nA"],
                        state["nB"], state["result"], state["workspace"])
    return {"nA": state["nA"], "nB": state["nB"], "result": state["result"]}


def _checkpoint(sim, case):
    """The raw state of a simulation as its values: deviations [direction][site][component] and, in 16-bit
    storage, the density deviations they refer to."""
    raw = sim.state()
    if ELEM[case["storage"]] != 2:
        return {"g": raw.view(DTYPE[case["storage"]])}
    n = 2 * 2 * sim.Q * sim.N
    return {"g": raw[:n].view(DTYPE[case["storage"]]), "ref": raw[n:].view(torch.float32)}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Every time step reads and writes the state once (the state of one step is the next one's input); the
    reads and writes of a pass's results come on top."""
    Q = 9 if case.get("lattice") == "d2q9" else 19
    site = 2 * Q * ELEM[case["storage"]] + (8 if ELEM[case["storage"]] == 2 else 0)  # bytes of one site's state
    sites = sum(m[0] * m[1] * m[2] for m in _members(case))
    nsteps = case.get("nsteps", 2) if case["kind"] != "check" else 2
    nbytes = sites * site * 2 * nsteps
    flops = sites * nsteps * (600 if Q == 19 else 280)
    if case["kind"] in ("steps", "sweep"):
        nbytes += 2 * sites * site  # the checkpoint: state read, copy written
    elif case["kind"] == "check":
        nbytes += sites * (site + 2 * 24)  # state read, previous velocity read and replaced
        flops += sites * 300
    elif case["kind"] == "tension":
        nbytes += sites * site
        flops += sites * 500
    elif case["kind"] == "fields":
        nbytes += sites * (site + 16 + 24 + 2 * 24)  # state read; densities, velocity written; previous velocity
        flops += sites * 400
    else:
        nbytes += sites * (2 * 16 + site + 2 * 16)  # host densities in and out (also over the link), first state
        flops += sites * 500
    return {"bytes": float(nbytes), "flops": float(flops)}


# ------------------------------------------------------------------ the method in FP64
_D3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
       (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1)]
_D2 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]


def _shift(a, v):
    """a(x + v) of a periodic field [z, y, x]."""
    return torch.roll(a, (-v[2], -v[1], -v[0]), (0, 1, 2)) if any(v) else a


class _Method:
    """One lattice in FP64: arriving populations f[J][i], advanced by whole-array shifts."""

    def __init__(self, case, m, seed):
        self.G, self.Gs, psi, _ = _couplings(m[3])
        self.psi_exp = psi == B.SC_PSI_EXP
        self.tau = case.get("tau", 1.0)
        d2 = case.get("lattice") == "d2q9"
        self.c = _D2 if d2 else _D3
        w = (4 / 9, 1 / 9, 1 / 36) if d2 else (1 / 3, 1 / 18, 1 / 36)
        self.w = [w[sum(x * x for x in c)] for c in self.c]
        if case.get("stencil") == "e6":
            W = {1: 2 / 15, 2: 1 / 15, 3: 1 / 60, 4: 1 / 120}
            self.force = [(v, W[q]) for v in itertools.product((-2, -1, 0, 1, 2), repeat=3)
                          for q in [sum(x * x for x in v)] if q in W]
        else:
            self.force = [(c, 3 * w) for c, w in zip(self.c[1:], self.w[1:])]
        self.n0 = _densities(m, seed)
        self.nbar = [float(n.mean()) for n in self.n0]
        self.f = [[w * n for w in self.w] for n in self.n0]
        self.post = self.n_at = None

    def _n(self):
        return [sum(f) for f in self.f]

    def _psi(self, n):
        return torch.exp(-1.0 / n) if self.psi_exp else n

    def _grad(self, a):
        g = [0.0, 0.0, 0.0]
        for v, W in self.force:
            s = _shift(a, v)
            for k in range(3):
                if v[k]:
                    g[k] = g[k] + (W * v[k]) * s
        return [x if torch.is_tensor(x) else torch.zeros_like(a) for x in g]

    def moments(self):
        n = self._n()
        grads, F = [self._grad(a) for a in n], []
        for J in (0, 1):
            Fj = [-self.G / 3 * n[J] * g for g in grads[1 - J]]
            if self.Gs[J]:
                p = self._psi(n[J])
                Fj = [a - self.Gs[J] / 3 * p * g for a, g in zip(Fj, self._grad(p))]
            F.append(Fj)
        u = []
        for k in range(3):
            j = sum(c[k] * f for J in (0, 1) for c, f in zip(self.c, self.f[J]) if c[k])
            u.append((j + 0.5 * (F[0][k] + F[1][k])) / (n[0] + n[1]))
        return n, u, F

    def step(self, count):
        for _ in range(count):
            n, u, F = self.moments()
            uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
            post = []
            for J in (0, 1):
                uF = u[0] * F[J][0] + u[1] * F[J][1] + u[2] * F[J][2]
                row = []
                for i, (c, w) in enumerate(zip(self.c, self.w)):
                    cu = sum(c[k] * u[k] for k in range(3) if c[k]) if any(c) else torch.zeros_like(uu)
                    cF = sum(c[k] * F[J][k] for k in range(3) if c[k]) if any(c) else torch.zeros_like(uu)
                    feq = w * n[J] * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
                    Fi = w * (3 * (cF - uF) + 9 * cu * cF)
                    row.append(self.f[J][i] + (feq - self.f[J][i]) / self.tau + (1 - 0.5 / self.tau) * Fi)
                post.append(row)
            self.f = [[_shift(g, tuple(-x for x in c)) for g, c in zip(row, self.c)] for row in post]
            self.post, self.n_at = post, n

    def checkpoint(self, case):
        lay = lambda pair: torch.stack([x.reshape(-1) for x in pair], -1).reshape(-1)  # noqa: E731  [site][J]
        if ELEM[case["storage"]] != 2:
            return {"g": torch.cat([lay([self.post[J][i] - w * self.nbar[J] for J in (0, 1)])
                                    for i, w in enumerate(self.w)])}
        g = None if case["storage"] == "f16" else torch.cat(
            [lay([self.post[J][i] - w * self.n_at[J] for J in (0, 1)]) for i, w in enumerate(self.w)])
        return {"g": g, "ref": lay([self.n_at[J] - self.nbar[J] for J in (0, 1)])}  # f16: scaled by a power of two

    def pressure(self):
        """The lattice pressure tensor {xx, yy, zz, xy, xz, yz} of every site."""
        n = self._n()
        psi = [self._psi(a) for a in n]
        idx = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]
        C = []
        for a in n + psi:
            s = [(v, W, _shift(a, v)) for v, W in self.force]
            C.append([sum((W * v[p] * v[q]) * x for v, W, x in s if v[p] * v[q]) + torch.zeros_like(a) for p, q in idx])
        P = []
        for k, (p, q) in enumerate(idx):
            t = (n[0] + n[1]) / 3 if p == q else 0.0
            P.append(t + (self.G * (n[0] * C[1][k] + n[1] * C[0][k]) + self.Gs[0] * psi[0] * C[2][k]
                          + self.Gs[1] * psi[1] * C[3][k]) / 6)
        return n, psi, P

    def bulk(self, n, psi, x, y, z):
        a, b, p, q = (float(t[z, y, x]) for t in (*n, *psi))
        return (a + b) / 3 + (self.G * a * b + 0.5 * self.Gs[0] * p * p + 0.5 * self.Gs[1] * q * q) / 3

    def tension(self, bin_width=0.5):
        """Radial profile rows and (dP, C, R_s, sigma_s, R_grid, sigma_grid, P_in, P_out)."""
        n, psi, P = self.pressure()
        nz, ny, nx = n[0].shape
        nbins = int(min(nx, ny, nz) / 2 / bin_width)
        d = []
        for k, L in enumerate((nx, ny, nz)):
            a = torch.arange(L, dtype=torch.float64, device=DEV) - L // 2
            a = a - L * torch.floor(a / L + 0.5)
            d.append(a.reshape([-1 if j == 2 - k else 1 for j in range(3)]).expand(nz, ny, nx))
        r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        e = [x / torch.where(r > 0, r, 1.0) for x in d]
        tr = P[0] + P[1] + P[2]
        PN = sum(e[k] * e[k] * P[k] for k in range(3)) + 2 * (e[0] * e[1] * P[3] + e[0] * e[2] * P[4] + e[1] * e[2] * P[5])
        PN = torch.where(r > 0, PN, tr / 3)
        PT = torch.where(r > 0, (tr - PN) / 2, tr / 3)
        b = torch.floor(r / bin_width).long().reshape(-1)
        keep = b < nbins
        rows = torch.zeros(nbins, 6, dtype=torch.float64, device=DEV)
        for k, v in enumerate((r, PN, PT, n[0], n[1], torch.ones_like(r))):
            rows[:, k] = torch.zeros(nbins, dtype=torch.float64, device=DEV).index_add_(0, b[keep], v.reshape(-1)[keep])
        rows[:, :5] = rows[:, :5] / rows[:, 5:].clamp(min=1)
        full = rows[rows[:, 5] > 0]
        x, f = full[:, 0], full[:, 0] ** 2 * full[:, 2]
        T = float((0.5 * (f[1:] + f[:-1]) * (x[1:] - x[:-1])).sum())
        Pin, Pout = self.bulk(n, psi, nx // 2, ny // 2, nz // 2), self.bulk(n, psi, nx - 1, ny - 1, nz - 1)
        dP, C = Pin - Pout, Pout * float(x[-1]) ** 3 / 3 - T
        Rs = math.copysign(abs(6 * C / dP) ** (1 / 3), 6 * C / dP)
        h, count = 0.01, int(math.floor((nbins * bin_width - 0.01) / 0.01 + 0.5)) + 1
        R = 0.01 + h * torch.arange(count, dtype=torch.float64)
        s = dP * R / 3 + C / (R * R)
        k = min(max(int(s.argmin()), 1), count - 2)
        y0, y1, y2 = (float(s[k + j]) for j in (-1, 0, 1))
        off = 0.5 * (y0 - y2) / (y0 - 2 * y1 + y2)
        return rows, torch.tensor([dP, C, Rs, 0.5 * dP * Rs, 0.01 + (k + off) * h, y1 - 0.25 * (y0 - y2) * off, Pin, Pout],
                                  dtype=torch.float64)


def exact(case, seed):
    ms = _members(case)
    if sum(m[0] * m[1] * m[2] for m in ms) * (case.get("nsteps", 2) + 8) > 1.2e9:
        return None
    kind, out = case["kind"], []
    for k, m in enumerate(ms):
        s = _Method(case, m, seed * 1009 + 31 * k)
        if kind in ("steps", "sweep"):
            s.step(case["nsteps"])
            out.append(s.checkpoint(case))
        elif kind == "check":
            u0 = s.moments()[1]
            s.step(2)
            n, u, _ = s.moments()
            psi = [s._psi(a) for a in n]
            dp = s.bulk(n, psi, m[0] // 2, m[1] // 2, m[2] // 2) - s.bulk(n, psi, m[0] - 1, m[1] - 1, m[2] - 1)
            out.append((dp, sum(float((a - b).abs().mean()) for a, b in zip(u, u0)),
                        torch.stack([a.reshape(-1) for a in u])))
        elif kind == "fields":
            u0 = s.moments()[1]
            s.step(case["nsteps"])
            n, u, _ = s.moments()
            j = [sum(float((c[a] * f).sum()) for J in (0, 1) for c, f in zip(s.c, s.f[J]) if c[a]) for a in range(3)]
            w = n[0] - 0.05
            M = float(w.sum())
            X = [float((w * torch.arange(L, dtype=torch.float64, device=DEV).reshape([-1 if q == 2 - a else 1 for q in range(3)])).sum()) / M
                 for a, L in enumerate(m[:3])]
            vec = lambda *v: torch.tensor(v, dtype=torch.float64)  # noqa: E731
            return {"nA": n[0].reshape(-1), "nB": n[1].reshape(-1), "u": torch.stack([a.reshape(-1) for a in u]),
                    "mass": vec(float(n[0].sum()), float(n[1].sum())),
                    "momentum": None if max(map(abs, j)) < 1e-6 else vec(*j),
                    "dU": vec(sum(float((a - b).abs().mean()) for a, b in zip(u, u0))), "centre": vec(*X, M)}
        else:
            s.step(case["nsteps"])
            if case["shape"] == "slab":
                n, psi, P = s.pressure()
                nz = m[2]
                mean = lambda a: a.reshape(nz, -1).mean(1)  # noqa: E731
                z = torch.arange(nz, dtype=torch.float64, device=DEV)
                rows = torch.stack([z, mean(P[2]), mean(0.5 * (P[0] + P[1])), mean(n[0]), mean(n[1]),
                                    torch.full_like(z, m[0] * m[1])], -1)
                return {"rows": rows, "result": (rows[nz // 2:, 1] - rows[nz // 2:, 2]).sum().reshape(1)}
            rows, res = s.tension()
            if kind == "tension":
                return {"rows": rows, "result": res}
            n = s._n()
            return {"nA": n[0].reshape(-1), "nB": n[1].reshape(-1), "result": res}
    if kind == "check":
        return {"dP": torch.tensor([o[0] for o in out], dtype=torch.float64),
                "dU": torch.tensor([o[1] for o in out], dtype=torch.float64), "u": [o[2] for o in out]}
    return out if "set" in case else out[0]
