"""What this library is used for, as measurable cases.

A case is a simulation that a program has set up (boxes with their parameters,
fields and launch mode) and ONE pass advances it by `steps` time steps, with
the spectra sampled on the way, and reads the results back through the public
API: psi and the velocity whole, the conserved totals, <u^2>, the per-mode mean
squares and the spectra.  Passes continue one another, as a run does between
its reads.

The fields are kept in single precision on the device, so a program that keeps
the results keeps them in single precision: `run` returns them so (the FP16
storage's velocity, which carries the populations' 16-bit rounding, as float16).

`exact` is the same scheme in plain torch, in 64 bits.
"""
import functools
import math

import numpy as np
import torch

import paper_1104_0078_gb300 as F

# Free energies and fluids of the workloads: (A, B, K, M, tau).
FREE_ENERGY = {
    "bulk": dict(A=0.05, B=0.0, K=0.04, M=0.1, tau=0.8),            # equilibrium fluctuations, 3D
    "bulk2d": dict(A=0.05, B=0.0, K=0.04, M=0.1, tau=1.0),          # the same in 2D
    "fluct15": dict(A=0.625, B=0.0, K=0.0, M=0.095, tau=1.1),       # the paper's own D3Q15 run
    "quench": dict(A=-0.0625, B=0.0625, K=0.04, M=0.1, tau=0.8),    # spinodal decomposition
    "capillary": dict(A=-0.05, B=0.05, K=0.2, M=0.1, tau=0.45),     # the paper's interfaces
}

DEFAULTS = dict(dim=3, q=19, nx=64, ny=64, nz=64, sizes="", nrep=1, energy="bulk", kT=1e-5, scheme="fv",
                integrator="heun", force="matched", lap="so", f16=False, mode="plain", tune=False, steps=50,
                every=0, mask=1, kmax=0, modes=False, start="noise")

SCHEME = {"fd": F.FLB_FD, "fv": F.FLB_FV, "naive": F.FLB_NAIVE}
INTEGRATOR = {"euler": F.FLB_EULER, "heun": F.FLB_HEUN, "rk4": F.FLB_RK4}
FORCE = {"matched": F.FLB_FORCE_MATCHED, "cd": F.FLB_FORCE_CD, "fv": F.FLB_FORCE_FV, "stress": F.FLB_FORCE_STRESS}
LAP = {"so": F.FLB_LAP_SO, "cd": F.FLB_LAP_CD, "pk": F.FLB_LAP_PK, "lb": F.FLB_LAP_LB}
MODE = {"plain": F.FLB_MODE_PLAIN, "batched": F.FLB_MODE_BATCHED, "persistent": F.FLB_MODE_PERSISTENT}


def listed():
    return [
        # The 2D bulk workload: equilibrium fluctuations on the smallest box of the tests, spectrum
        # and mode variances sampled.  A step is a few microseconds of work: launches and latency.
        dict(name="bulk_2d_64", dim=2, q=9, nx=64, ny=64, nz=1, energy="bulk2d", kT=1e-4, scheme="fd", steps=200,
             every=20, modes=True, start="fluct"),
        # 2D coarsening, a large planar run: bandwidth.
        dict(name="quench_2d_2048", dim=2, q=9, nx=2048, ny=2048, nz=1, energy="quench", kT=1e-5, scheme="fd",
             steps=200, every=50, kmax=16),
        # The paper's order-parameter fluctuation run: D3Q15 32^3, finite differences, the whole spectrum.
        dict(name="fluct_d3q15_32", q=15, nx=32, ny=32, nz=32, energy="fluct15", kT=1.0 / 3000.0, scheme="fd",
             steps=100, every=10, modes=True, start="fluct"),
        # The 3D bulk workload as the statistics runs drive it: one 64^3 box, no tuning.
        dict(name="bulk_3d_64", nx=64, ny=64, nz=64, kT=1e-5, steps=100, every=25, modes=True, start="fluct"),
        # An odd box in half-precision storage, coarsening.
        dict(name="ragged_f16", nx=101, ny=75, nz=53, energy="quench", kT=1e-5, f16=True, steps=100, every=20, kmax=12),
        # The slab workload: two interfaces, capillary height spectrum and psi spectrum.
        dict(name="slab_256x64", nx=256, ny=256, nz=64, energy="capillary", kT=1.0 / 3000.0, steps=80, every=10, mask=3,
             kmax=8, start="slab"),
        # The headline run: 512^3 spinodal quench, S(q) every 10 steps, tuned as the README shows.
        dict(name="quench_512", nx=512, ny=512, nz=512, energy="quench", kT=1e-5, steps=50, every=10, kmax=8,
             tune=True),
        # The finite-difference scheme on a middle-sized box.
        dict(name="quench_fd_160", nx=160, ny=160, nz=160, energy="quench", kT=1e-5, scheme="fd", steps=80, tune=True),
        # The uneven ensemble: 256 replicas from 16^3 to 48^3 in one handle, batched.
        dict(name="ensemble_256", sizes="16,24,32,48", nrep=256, kT=5e-5, mode="batched", tune=True, steps=100,
             start="fluct"),
        # 25 replicas of the paper's D3Q15 fluctuation box, all steps in one cooperative launch.
        dict(name="ensemble_d3q15", q=15, sizes="32", nrep=25, energy="fluct15", kT=1.0 / 3000.0, mode="persistent",
             tune=True, steps=100, start="fluct"),
        # Fourth-order integration with the momentum-conserving stress force.
        dict(name="rk4_stress_128", nx=128, ny=128, nz=128, energy="quench", kT=1e-5, integrator="rk4", force="stress",
             steps=80, tune=True),
        # A stencil study: finite volumes with the Patra-Karttunen Laplacian (per-site kernels).
        dict(name="stencil_pk_96", nx=96, ny=96, nz=96, kT=1e-5, lap="pk", steps=100, start="fluct"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more run of the kinds listed: any lattice, scheme, size and aspect."""
    kind = rng.choice(["planar", "box", "box", "box", "study", "replicas"])
    if kind == "planar":
        nx, ny = _log_int(rng, 40, 3000), _log_int(rng, 40, 3000)
        n = nx * ny
        energy = rng.choice(["bulk2d", "quench"])
        return dict(dim=2, q=9, nx=nx, ny=ny, nz=1, energy=energy, kT=10.0 ** rng.uniform(-5.0, -4.0),
                    scheme=rng.choice(["fd", "fv"]), integrator=rng.choice(["heun", "heun", "euler", "rk4"]),
                    f16=rng.random() < 0.2, steps=max(20, min(200, 300_000_000 // n)), every=20, kmax=rng.randint(4, 16),
                    start="fluct" if energy == "bulk2d" else "noise")
    if kind in ("box", "study"):
        edge = math.exp(rng.uniform(math.log(16), math.log(320 if kind == "box" else 128)))
        nx, ny, nz = (max(8, int(round(edge * math.exp(rng.uniform(-0.4, 0.4))))) for _ in range(3))
        n = nx * ny * nz
        # the central-difference Laplacian is unstable with the capillary K
        energy = rng.choice(["bulk", "quench", "capillary"] if kind == "box" else ["bulk", "quench"])
        c = dict(q=rng.choice([19, 19, 15]), nx=nx, ny=ny, nz=nz, energy=energy, kT=10.0 ** rng.uniform(-5.0, -4.0),
                 steps=max(10, min(100, 300_000_000 // n)), every=10, kmax=rng.randint(4, 12),
                 start={"bulk": "fluct", "quench": "noise", "capillary": "slab"}[energy])
        if kind == "study":
            scheme = rng.choice(["fv", "naive", "fd"])
            return dict(c, scheme=scheme, lap=rng.choice(["cd", "pk", "lb"]), integrator=rng.choice(["heun", "euler"]))
        c.update(scheme=rng.choice(["fv", "fv", "fd"]), integrator=rng.choice(["heun", "heun", "heun", "euler", "rk4"]),
                 f16=rng.random() < 0.25, tune=rng.random() < 0.3)
        if rng.random() < 0.15:
            c["force"] = "stress"
        return c
    edges = ",".join(str(rng.randint(12, 52)) for _ in range(rng.choice([1, 2, 4])))
    q = rng.choice([19, 19, 15])
    return dict(q=q, sizes=edges, nrep=_log_int(rng, 8, 160), energy=rng.choice(["bulk", "quench"]),
                kT=10.0 ** rng.uniform(-5.0, -4.0), integrator=rng.choice(["heun", "heun", "euler"]),
                mode=rng.choice(["batched", "batched", "persistent"]), steps=rng.randint(30, 60), start="noise")


# ---- the runs --------------------------------------------------------------------------------------------------------


def _full(case):
    return {**DEFAULTS, **case}


def _boxes(c):
    """The edges of every replica: the listed sizes in equal parts, or the one box."""
    if not c["sizes"]:
        return [(c["nx"], c["ny"], c["nz"])]
    edges = [int(e) for e in str(c["sizes"]).split(",")]
    per = [c["nrep"] // len(edges) + (k < c["nrep"] % len(edges)) for k in range(len(edges))]
    return [(e, e, e) for e, k in zip(edges, per) for _ in range(k)]


def _box_kT(c, r):
    """Replicas run over a range of temperatures around the case's own."""
    return c["kT"] * (0.2 + 1.6 * ((r * 0.6180339887) % 1.0)) if c["sizes"] else c["kT"]


def _box_seed(seed, r):
    return (int(seed) * 1_000_003 + 7919 * r + 1) & 0xFFFFFFFF


def _start_fields(c, box, kT, seed):
    """psi and u of one replica at step 0, single-precision values, made on the device."""
    nx, ny, nz = box
    d = c["dim"]
    e = FREE_ENERGY[c["energy"]]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev)
    g.manual_seed(_box_seed(seed, 0))
    shape = (nz, ny, nx)
    if c["start"] == "slab":
        z = torch.arange(nz, device=dev, dtype=torch.float64)
        ell, pb = math.sqrt(2.0 * e["K"] / abs(e["A"])), math.sqrt(abs(e["A"]) / max(e["B"], 1e-9))
        prof = pb * torch.tanh((z - 0.25 * nz) / ell) * torch.tanh((0.75 * nz - z) / ell)
        psi = prof.float()[:, None, None] + 0.01 * torch.randn(shape, generator=g, device=dev)
    elif c["start"] == "fluct":
        psi = math.sqrt(kT / e["A"]) * torch.randn(shape, generator=g, device=dev)
    else:
        psi = 0.02 * torch.rand(shape, generator=g, device=dev) - 0.01
    u = math.sqrt(kT) * torch.randn((d,) + shape, generator=g, device=dev)
    return psi, u


def prepare(case, seed):
    c = _full(case)
    e = FREE_ENERGY[c["energy"]]
    boxes = _boxes(c)
    params = [
        F.flb_params_default(dim=c["dim"], q=c["q"], nx=b[0], ny=b[1], nz=b[2], tau=e["tau"], kT=_box_kT(c, r), A=e["A"],
                             B=e["B"], K=e["K"], M=e["M"], psi_scheme=SCHEME[c["scheme"]],
                             integrator=INTEGRATOR[c["integrator"]],
                             storage=F.FLB_F16_DEV if c["f16"] else F.FLB_F32_DEV, seed=_box_seed(seed, r),
                             sq_kmax=c["kmax"], force_grad=FORCE[c["force"]], laplacian=LAP[c["lap"]],
                             init=F.FLB_INIT_USER)
        for r, b in enumerate(boxes)
    ]
    s = F.Solver(params)
    for r, b in enumerate(boxes):
        psi, u = _start_fields(c, b, params[r].kT, seed + 31 * r)
        s.set_fields(rep=r, psi=psi.double().cpu().numpy(), u=u.double().cpu().numpy())
    if c["every"]:
        s.set_sampling(c["every"], c["mask"])
    s.set_mode(MODE[c["mode"]])
    if c["tune"]:
        s.autotune()
    n = sum(x * y * z for x, y, z in boxes)  # where the fields are kept once read
    return {"solver": s, "case": c, "psi": torch.zeros(n), "u": torch.zeros(c["dim"] * n)}


def _f32(a):
    return torch.from_numpy(a).float()


def run(state):
    s, c = state["solver"], state["case"]
    s.step(c["steps"])
    psi, u, at, d = state["psi"], state["u"], 0, c["dim"]
    for r in range(len(s.params)):
        p, v = s.get_psi_u(r)
        psi[at:at + p.size].copy_(torch.from_numpy(p))
        u[d * at:d * (at + p.size)].copy_(torch.from_numpy(v).reshape(-1))
        at += p.size
    totals, u2 = [], []
    for r in range(min(len(s.params), 8)):
        t, w, _ = s.moments(r)
        totals.append(_f32(t))
        u2.append(_f32(w))
    out = {"psi": psi, "u": u, "totals": torch.cat(totals), "u2": torch.cat(u2)}
    if c["f16"]:
        out["u"] = out["u"].half()
    if c["modes"]:
        out["modes"] = _f32(s.mode_variances(0))
    if c["every"]:
        out["sq"] = _f32(s.structure_factor(0)[0])
        if c["mask"] & 2:
            out["sq_height"] = _f32(s.structure_factor(0, F.FLB_SQ_HEIGHT)[0])
    return out


def work(case):
    """Populations, psi and u in and out once a step; u is what a step hands to a read, psi and the
    populations are the state.  Arithmetic: collision (about 20 q), normals (about 40 each, q - dim - 1 of
    the fluid and those of psi) and the psi stages (about 120 each in 3D, 60 in 2D) per site and step."""
    c = _full(case)
    n = sum(x * y * z for x, y, z in _boxes(c)) * c["steps"]
    pop = c["q"] * (2 if c["f16"] else 4)
    stages = {"euler": 1, "heun": 2, "rk4": 4}[c["integrator"]]
    normals = c["q"] - c["dim"] - 1
    normals += (13 if c["dim"] == 3 else 4) if c["scheme"] == "fd" else c["dim"]
    return {"bytes": float(n * (2 * pop + 8)),
            "flops": float(n * (20 * c["q"] + 40 * normals + stages * (120 if c["dim"] == 3 else 60)))}


# ---- the same scheme in 64 bits --------------------------------------------------------------------------------------

C9 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]
C15 = C9[:5] + [(0, 0, 1), (0, 0, -1), (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1),
                (1, -1, -1), (-1, 1, 1)]
C19 = C9[:5] + [(0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1),
                (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
LATTICE = {9: (C9, (4 / 9, 1 / 9, 1 / 36, 0)), 15: (C15, (2 / 9, 1 / 9, 0, 1 / 72)), 19: (C19, (1 / 3, 1 / 18, 1 / 36, 0))}
LINKS = {2: [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)],
         3: [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1),
             (1, 1, 1), (1, 1, -1), (1, -1, 1), (1, -1, -1)]}
LAP_CLASS = {(3, "so"): (6 / 22, 3 / 22, 1 / 22), (3, "cd"): (1.0, 0.0, 0.0), (3, "pk"): (14 / 30, 3 / 30, 1 / 30),
             (3, "lb"): (1 / 9, 1 / 9, 1 / 9), (2, "so"): (0.5, 0.25, 0.0), (2, "cd"): (1.0, 0.0, 0.0)}


def _at(a, c):
    """The field a at r + c (x is the last axis)."""
    return torch.roll(a, (-c[2], -c[1], -c[0]), (-3, -2, -1)) if any(c) else a


@functools.lru_cache(maxsize=None)
def _basis(dim, q):
    """Gram-Schmidt moment basis under sum_i w_i a_i b_i on the ordered monomials, and its norms."""
    cs, wc = LATTICE[q]
    w = np.array([wc[sum(map(abs, v))] for v in cs])
    x, y, z = np.array(cs, dtype=np.float64).T
    c2 = x * x + y * y + z * z
    one = np.ones(q)
    if dim == 2:
        mono = [one, x, y, c2, x * x - y * y, x * y, c2 * x, c2 * y, c2 * c2]
    else:
        mono = [one, x, y, z, c2, 3 * x * x - c2, y * y - z * z, x * y, y * z, z * x, c2 * x, c2 * y, c2 * z]
        mono += ([x * y * z, c2 * c2] if q == 15 else
                 [x * (y * y - z * z), y * (z * z - x * x), z * (x * x - y * y), c2 * c2, c2 * (3 * x * x - c2),
                  c2 * (y * y - z * z)])
    E = []
    for m in mono:
        for e in E:
            m = m - (w * m * e).sum() / (w * e * e).sum() * e
        E.append(m)
    E = np.array(E)
    return w, E, (w * E * E).sum(1)


class Reference:
    """R boxes of one size side by side: fields are (R, nz, ny, nx) in 64 bits."""

    def __init__(self, c, box, kTs, seeds, fields, dev):
        self.c, self.box, self.dev = c, box, dev
        self.e = FREE_ENERGY[c["energy"]]
        col = lambda v, t: torch.tensor(v, dtype=t, device=dev).reshape(-1, 1, 1, 1)  # noqa: E731
        self.kT = col(kTs, torch.float64)
        self.key = (col([s & 0xFFFFFFFF for s in seeds], torch.int64), col([s >> 32 for s in seeds], torch.int64))
        nx, ny, nz = box
        self.site = torch.arange(nx * ny * nz, device=dev, dtype=torch.int64).reshape(1, nz, ny, nx)
        self.psi = torch.stack([f[0] for f in fields]).double()
        self.u = [torch.stack([f[1][a] for f in fields]).double() for a in range(c["dim"])]
        self.w, self.E, self.b = _basis(c["dim"], c["q"])
        self.vel = LATTICE[c["q"]][0]
        self.step = 0
        u2 = sum(v * v for v in self.u)
        self.f = []  # deviations from w_i of the streamed populations
        for w, v in zip(self.w, self.vel):
            cu = sum(v[a] * self.u[a] for a in range(c["dim"]))
            self.f.append(w * (3.0 * cu + 4.5 * cu * cu - 1.5 * u2))

    def normals(self, stream, n):
        out = []
        for block in range((n + 7) // 8):
            x = [self.site, torch.full_like(self.site, self.step & 0xFFFFFFFF),
                 torch.full_like(self.site, (stream << 16) | block), torch.full_like(self.site, self.step >> 32)]
            k0, k1 = self.key
            for _ in range(10):
                p0, p1 = 0xD2511F53 * x[0], 0xCD9E8D57 * x[2]
                x = [((p1 >> 32) & 0xFFFFFFFF) ^ x[1] ^ k0, p1 & 0xFFFFFFFF, ((p0 >> 32) & 0xFFFFFFFF) ^ x[3] ^ k1,
                     p0 & 0xFFFFFFFF]
                k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
            for k in range(4):
                if len(out) < n:
                    r = torch.sqrt(-2.0 * torch.log(((x[k] >> 12).double() + 0.5) / 1048576.0))
                    t = ((x[k] & 0xFFF).double() + 0.5) * (2.0 * math.pi / 4096.0)
                    out += [r * torch.cos(t), r * torch.sin(t)]
        return out[:n]

    def lap(self, a, kind):
        cw = LAP_CLASS[self.c["dim"], kind]
        zs = (-1, 0, 1) if self.c["dim"] == 3 else (0,)
        near = [0.0, 0.0, 0.0]
        for v in ((x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in zs):
            k = sum(map(abs, v))
            if k and cw[k - 1]:
                near[k - 1] = near[k - 1] + _at(a, v)
        count = (6, 12, 8) if self.c["dim"] == 3 else (4, 4, 0)
        return sum(w * s for w, s in zip(cw, near)) - sum(w * k for w, k in zip(cw, count)) * a

    def mu(self, psi):
        e = self.e
        return e["A"] * psi + e["B"] * psi ** 3 - e["K"] * self.lap(psi, self.c["lap"])

    def cd(self, a, axis):
        v = tuple(int(k == axis) for k in range(3))
        return 0.5 * (_at(a, v) - _at(a, tuple(-k for k in v)))

    def fv_grad(self, a):
        g = [0.0] * self.c["dim"]
        for w, v in zip(self.w[1:], self.vel[1:]):
            m = (3.0 * w) * _at(a, v)
            for k in range(self.c["dim"]):
                if v[k]:
                    g[k] = g[k] + v[k] * m
        return g

    def fv_div(self, J):
        """(2/c_s^2) sum_i w_i c_i . (J(r) + J(r + c_i))/2; the J(r) terms cancel over the lattice."""
        out = 0.0
        for w, v in zip(self.w[1:], self.vel[1:]):
            out = out + (3.0 * w) * _at(sum(v[k] * J[k] for k in range(self.c["dim"]) if v[k]), v)
        return out

    def force(self):
        c, e, d, psi = self.c, self.e, self.c["dim"], self.psi
        if c["force"] == "stress":
            g = [self.cd(psi, a) for a in range(d)]
            p2 = psi * psi
            iso = 0.5 * e["A"] * p2 + 0.75 * e["B"] * p2 * p2 - e["K"] * psi * self.lap(psi, c["lap"])
            iso = iso - 0.5 * e["K"] * sum(x * x for x in g)
            return [-sum(self.cd(e["K"] * g[a] * g[b] + (iso if a == b else 0.0), b) for b in range(d)) for a in range(d)]
        mu = self.mu(psi)
        fv = c["force"] == "fv" or (c["force"] == "matched" and c["scheme"] == "fv")
        grad = self.fv_grad(mu) if fv else [self.cd(mu, a) for a in range(d)]
        return [-psi * x for x in grad]

    def fluid(self):
        c, d, q = self.c, self.c["dim"], self.c["q"]
        Fv = self.force()
        f = torch.stack(self.f).reshape(q, -1)
        flat = lambda a: a.reshape(-1)  # noqa: E731
        mat = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=self.dev)  # noqa: E731
        cv = np.array(self.vel, dtype=np.float64)
        pairs = [(a, b) for a in range(d) for b in range(a, d)]
        Q = [cv[:, a] * cv[:, b] - (1.0 / 3.0 if a == b else 0.0) for a, b in pairs]
        mom = mat(np.array([np.ones(q)] + [cv[:, a] for a in range(d)] + Q)) @ f
        drho, j, S = mom[0], mom[1:1 + d], dict(zip(pairs, mom[1 + d:]))
        Fl = [flat(x) for x in Fv]
        rho = 1.0 + drho
        v = [(j[a] + 0.5 * Fl[a]) / rho for a in range(d)]
        om = 1.0 / (self.e["tau"] + 0.5)
        rows = [drho] + [j[a] + Fl[a] for a in range(d)]
        cols = [np.ones(q)] + [3.0 * cv[:, a] for a in range(d)]
        for k, (a, b) in enumerate(pairs):
            rows.append(S[a, b] + om * (rho * v[a] * v[b] - S[a, b]) + (1.0 - 0.5 * om) * (v[a] * Fl[b] + Fl[a] * v[b]))
            cols.append((4.5 if a == b else 9.0) * Q[k])
        G = self.normals(0, q - d - 1)
        amp = torch.sqrt(3.0 * rho * flat(self.kT.expand_as(self.psi)))
        for t, g in enumerate(G):
            k = d + 1 + t
            gam = 1.0 - om if t < len(pairs) else 0.0
            rows.append(amp * flat(g) * math.sqrt(self.b[k] * (1.0 - gam * gam)))
            cols.append(self.E[k] / self.b[k])
        del G, f, mom
        post = mat(self.w[:, None] * np.array(cols).T) @ torch.stack(rows)
        del rows
        shape = self.psi.shape
        self.f = [_at(post[i].reshape(shape), tuple(-k for k in self.vel[i])) for i in range(q)]
        del post
        drho = sum(self.f)
        self.u = [(sum(self.vel[i][a] * self.f[i] for i in range(q) if self.vel[i][a]) + 0.5 * Fv[a]) / (1.0 + drho)
                  for a in range(d)]

    def noise(self):
        """The noise of one psi step: the increment eta (FD, naive) or the node flux xi (FV)."""
        c, d = self.c, self.c["dim"]
        sd = torch.sqrt(2.0 * self.kT * self.e["M"])
        if c["scheme"] == "fd":
            cw, eta = LAP_CLASS[d, c["lap"]], 0.0
            for l, g in zip(LINKS[d], self.normals(1, len(LINKS[d]))):
                z = sd * math.sqrt(cw[sum(map(abs, l)) - 1]) * g
                eta = eta + (_at(z, tuple(-k for k in l)) - z)
            return eta
        xi = [sd * g for g in self.normals(1, d)]
        return xi if c["scheme"] == "fv" else sum(self.cd(xi[a], a) for a in range(d))

    def rhs(self, psi, noise):
        c, d = self.c, self.c["dim"]
        mu = self.mu(psi)
        if c["scheme"] == "fv":
            g = self.fv_grad(mu)
            return self.fv_div([self.e["M"] * g[a] - self.u[a] * psi + noise[a] for a in range(d)])
        return self.e["M"] * self.lap(mu, c["lap"]) - sum(self.cd(self.u[a] * psi, a) for a in range(d)) + noise

    def advance(self):
        self.fluid()
        p, n = self.psi, self.noise()
        k1 = self.rhs(p, n)
        kind = self.c["integrator"]
        if kind == "euler":
            self.psi = p + k1
        elif kind == "heun":
            self.psi = p + 0.5 * (k1 + self.rhs(p + k1, n))
        else:
            k2 = self.rhs(p + 0.5 * k1, n)
            k3 = self.rhs(p + 0.5 * k2, n)
            self.psi = p + (k1 + 2.0 * k2 + 2.0 * k3 + self.rhs(p + k3, n)) / 6.0
        self.step += 1

    def spectrum(self):
        """|psi~(q)|^2 of box 0 in the window of the case."""
        a = self.psi[0]
        s = torch.fft.fftn(a).abs().square() / a.numel()
        for axis, n in ((2, self.box[0]), (1, self.box[1]), (0, self.box[2])):
            k = self.c["kmax"]
            if 0 < k and 2 * k + 1 < n:
                s = torch.cat([s.narrow(axis, 0, k + 1), s.narrow(axis, n - k, k)], axis)
        return s.reshape(-1)


def exact(case, seed):
    c = _full(case)
    boxes = _boxes(c)
    sites = sum(x * y * z for x, y, z in boxes)
    if sites * c["steps"] > 1_000_000_000:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    groups = {}
    for r, b in enumerate(boxes):
        groups.setdefault(b, []).append(r)
    psi, u, totals, u2, sq, modes = ([None] * len(boxes) for _ in range(6))
    for b, reps in groups.items():
        kTs = [_box_kT(c, r) for r in reps]
        m = Reference(c, b, kTs, [_box_seed(seed, r) for r in reps],
                      [_start_fields(c, b, kT, seed + 31 * r) for r, kT in zip(reps, kTs)], dev)
        samples, spec = 0, 0.0
        for _ in range(c["steps"]):
            m.advance()
            if c["every"] and m.step % c["every"] == 0 and reps[0] == 0:
                spec, samples = spec + m.spectrum(), samples + 1
        f = torch.stack(m.f)
        for k, r in enumerate(reps):
            psi[r], u[r] = m.psi[k].reshape(-1), torch.cat([x[k].reshape(-1) for x in m.u])
            if r < 8:
                n = float(b[0] * b[1] * b[2])
                fr = f[:, k].reshape(c["q"], -1)
                j = [sum(m.vel[i][a] * fr[i].sum() for i in range(c["q"])) for a in range(c["dim"])]
                totals[r] = torch.stack([n + fr.sum()] + j + [psi[r].sum()])
                u2[r] = torch.stack([x[k].square().mean() for x in m.u])
            if r == 0:
                sq[0] = spec / samples if samples else None
                E = torch.tensor(m.E, dtype=torch.float64, device=dev)
                modes[0] = (E @ f[:, 0].reshape(c["q"], -1)).square().mean(1)
    cat = lambda v: torch.cat([x for x in v if x is not None])  # noqa: E731
    out = {"psi": cat(psi), "u": cat(u), "totals": cat(totals), "u2": cat(u2)}
    if c["modes"]:
        out["modes"] = modes[0]
    if c["every"] and c["mask"] & 1:
        out["sq"] = sq[0]
    return out
