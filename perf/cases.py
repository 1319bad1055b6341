"""The work a user has this library do, as cases that can be timed and checked.

A pass is what a simulation program does between two looks at its fields: advance the state
by some timesteps, then read the macroscopic fields (rho^s, U and, where no component
vanishes, mu^s) into device tensors it keeps -- through `Simulation` and `Batch` as a
program calls them.  Batches and the whole job read their fields on the host, the only way
these calls offer.  FP64 runs keep FP64 fields; runs stored in FP32 or 16 bits keep their
snapshots in FP32.

The state moves on from pass to pass, as it does in a program.  Every start has a flow of a
few hundredths of the lattice speed, so that U is more than rounding, and compositions inside
the range where the method is stable for any number of passes.

`exact` is the method in 64 bits in plain torch: one generic update over (N, Q, z, y, x)
with rolls, written from the equations, sharing no code with the library.
"""
import math

import numpy as np
import torch

import paper_0704_3444_gb300 as mclb

PRECISION_BYTES = {"fp64": (8, 0), "fp32": (4, 0), "bf16": (2, 4), "fp16": (2, 4)}  # value, R
CAP = 2048 * 2048 * 5 * 50   # most sites * components * timesteps of a D2Q9 pass
CAP_CUBE = 192 * 192 * 192 * 3 * 15


def listed():
    return [
        # the smallest run of the method: a binary mixture separating on 64 x 64 in FP64; every
        # step is far shorter than a launch, so launches and latency are all there is
        dict(name="binary_64_fp64", kind="plane", n=2, nx=64, ny=64, precision="fp64", start="mixed",
             chi=2.2, tau=1.0, kappa=0.01, m0=1.0, steps=100),
        # the ordinary two-dimensional run: a phase-separated ternary on 256 x 256, FP32
        dict(name="ternary_256_fp32", kind="plane", n=3, nx=256, ny=256, precision="fp32",
             start="droplets", chi=2.4, tau=0.8, kappa=0.01, m0=1.0, steps=100),
        # a coupled or interactive program: one timestep per call, fields read after each, on an
        # odd four-component grid in FP16 storage
        dict(name="onestep_300x170_fp16", kind="plane", n=4, nx=300, ny=170, precision="fp16",
             start="mixed", chi=1.9, tau=0.9, kappa=0.01, m0=1.0, steps=1),
        # the headline workload: five components on 2048 x 2048, FP32 storage
        dict(name="n5_2048_fp32", kind="plane", n=5, nx=2048, ny=2048, precision="fp32",
             start="mixed", chi=0.0, tau=1.0, kappa=0.01, m0=1.0, steps=50),
        # the same in 16-bit shifted storage
        dict(name="n5_2048_bf16", kind="plane", n=5, nx=2048, ny=2048, precision="bf16",
             start="mixed", chi=0.0, tau=1.0, kappa=0.01, m0=1.0, steps=50),
        # the largest lattice of the workloads: polymer solution against non-solvent, 8192 x 2048
        dict(name="slab_8192x2048_fp32", kind="plane", n=3, nx=8192, ny=2048, precision="fp32",
             start="slab", chi=3.0, tau=1.0 / 0.9, kappa=0.01, m0=1.0, steps=20),
        # a ragged channel between solid walls, driven by a body force
        dict(name="channel_1000x333_fp32", kind="channel", n=3, nx=1000, ny=333, precision="fp32",
             start="mixed", chi=1.8, tau=0.8, kappa=0.01, m0=1.0, steps=60),
        # the polymer binary under the Gibbs-Duhem force form with the barycentric forcing
        # velocity, FP64 as the validation runs use it
        dict(name="polymer_160x96_fp64", kind="polymer", n=2, nx=160, ny=96, precision="fp64",
             start="layers", chi=0.9, tau=1.0 / 0.9, kappa=0.0, m0=10.0, steps=50),
        # a parameter sweep: independent binary and ternary lattices of uneven size in one batch
        dict(name="batch_48_fp32", kind="batch", count=48, lo=32, hi=512, precision="fp32", steps=200),
        # the paper's own experiment: a sweep of D1Q3 lines in FP64
        dict(name="lines_60x128_fp64", kind="lines", count=60, n=2, nx=128, precision="fp64", m0=1.0,
             gd=0, steps=2000),
        # three dimensions: a separating ternary on 192^3, FP32
        dict(name="cube_192_fp32", kind="cube", n=3, nx=192, ny=192, nz=192, precision="fp32",
             chi=2.6, tau=1.0 / 0.9, kappa=0.01, steps=15),
        # a whole job from host arrays to host results: upload, run, fields, sums and fit
        dict(name="job_512x384_fp32", kind="job", n=3, nx=512, ny=384, precision="fp32",
             start="droplets", chi=2.4, tau=0.8, kappa=0.01, m0=1.0, steps=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plane", "plane", "plane", "plane", "channel", "polymer", "batch", "lines",
                       "cube", "job"])
    if kind == "batch":
        lo = rng.randint(32, 64)
        return dict(kind=kind, count=rng.randint(8, 48), lo=lo, hi=rng.randint(lo + 32, 512),
                    precision=rng.choice(["fp32", "fp32", "bf16", "fp64"]), steps=rng.randint(20, 60))
    if kind == "lines":
        return dict(kind=kind, count=_log(rng, 4, 512), n=rng.randint(2, 3), nx=_log(rng, 48, 600),
                    precision=rng.choice(["fp64", "fp64", "fp32"]), m0=rng.choice([1.0, 1.0, 10.0]),
                    gd=rng.randint(0, 1), steps=_log(rng, 100, 800))
    if kind == "cube":
        n = rng.randint(2, 4)
        s = [_log(rng, 24, 200) for _ in range(3)]
        while s[0] * s[1] * s[2] * n > CAP_CUBE // 4:
            s = [max(24, v * 9 // 10) for v in s]
        prec = rng.choice(["fp32", "fp32", "fp64"])
        most = CAP_CUBE // (s[0] * s[1] * s[2] * n * (8 if prec == "fp64" else 1))
        return dict(kind=kind, n=n, nx=s[0], ny=s[1], nz=s[2], precision=prec,
                    chi=round(rng.uniform(1.5, 2.6), 2), tau=round(rng.uniform(0.7, 1.2), 3),
                    kappa=0.01, steps=max(1, min(rng.randint(2, 20), most)))
    n = rng.randint(2, 3) if kind in ("polymer", "job") else rng.randint(1, 6)
    prec = rng.choice({"plane": ["fp32", "fp32", "fp32", "bf16", "fp16", "fp64"],
                       "channel": ["fp32", "fp32", "bf16", "fp64"],
                       "polymer": ["fp64", "fp32"], "job": ["fp32", "fp64"]}[kind])
    top = {"plane": 4096, "channel": 2048, "polymer": 512, "job": 768}[kind]
    nx, ny = _log(rng, 40, top), _log(rng, 40, top)
    most = CAP // (n * nx * ny * (16 if prec == "fp64" else 1))
    if most < 1:
        nx, ny = nx // 3, ny // 3
        most = CAP // (n * nx * ny * 16)
    steps = 1 if kind == "plane" and rng.random() < 0.15 else max(1, min(_log(rng, 4, 120), most))
    start = "layers" if kind == "polymer" else "droplets" if n == 3 and rng.random() < 0.4 else "mixed"
    return dict(kind=kind, n=n, nx=nx, ny=ny, precision=prec, start=start,
                chi=0.9 if kind == "polymer" else round(rng.uniform(1.6, 2.4), 2),
                tau=round(rng.uniform(0.75, 1.2), 3), kappa=0.0 if kind == "polymer" else 0.01,
                m0=10.0 if kind == "polymer" else 1.0, steps=steps)


# ---------------------------------------------------------------- parameters and inputs

def _chi(case, seed):
    n = case["n"]
    chi = np.full((n, n), float(case["chi"]))
    if case["chi"] == 0.0:      # random symmetric in [0.8, 1.5] x the pair critical value 2
        r = np.random.RandomState(seed % (1 << 31))
        chi = 2.0 * r.uniform(0.8, 1.5, (n, n))
        chi = np.triu(chi, 1) + np.triu(chi, 1).T
    np.fill_diagonal(chi, 0.0)
    if case.get("start") == "slab":   # polymer, solvent, non-solvent
        chi[0, 1] = chi[1, 0] = 0.5
        chi[1, 2] = chi[2, 1] = 0.2
    return chi


def _params(case, seed):
    n, kind = case["n"], case["kind"]
    m = np.ones(n)
    m[0] = case.get("m0", 1.0)
    force = (2e-6, 0.0) if kind == "channel" else (1e-7, -5e-8, 2e-8) if kind == "cube" else (0.0, 0.0)
    return dict(ncomp=n, nx=case["nx"], ny=case["ny"], nz=case.get("nz", 1), tau=case["tau"],
                chi=_chi(case, seed), m=m, theta=1.0 / 3.0, kappa=case["kappa"], force=force,
                forcing_velocity=int(kind == "polymer"), force_form=int(kind == "polymer"),
                lattice="d3q19" if kind == "cube" else "d2q9", walls=int(kind == "channel"))


def _fields(case, seed, device):
    """rho (N, [nz,] ny, nx) and u (2 or 3, ...) in FP64 from the seed alone."""
    g = torch.Generator(device=device).manual_seed(seed)
    kw = dict(device=device, dtype=torch.float64)

    def rand(*shape):
        return torch.rand(*shape, generator=g, **kw)

    n, nx, ny, nz = case["n"], case["nx"], case["ny"], case.get("nz", 1)
    x = torch.arange(nx, **kw)[None, None, :]
    y = torch.arange(ny, **kw)[None, :, None]
    z = torch.arange(nz, **kw)[:, None, None]
    tp = 2.0 * math.pi
    ph = tp * rand(8)
    start = "cube" if case["kind"] == "cube" else case["start"]
    noise = 0.01 * (2.0 * rand(n, nz, ny, nx) - 1.0)
    noise -= noise.mean(0, keepdim=True)
    if start in ("mixed", "cube"):
        base = torch.full((n, 1, 1, 1), 1.0 / n, **kw)
        if n > 1:
            wave = 0.05 * torch.sin(tp * x / nx + ph[0]) * torch.cos(tp * y / ny + ph[1])
            noise[0] += wave
            noise[1] -= wave
        rho = base + noise
    elif start == "droplets":   # six discs of an A-rich phase in a B-rich matrix
        d = torch.zeros(1, ny, nx, **kw)
        r = rand(6, 3)
        for k in range(6):
            dx = (x - r[k, 0] * nx).abs()
            dy = (y - r[k, 1] * ny).abs()
            dist = torch.sqrt(torch.minimum(dx, nx - dx) ** 2 + torch.minimum(dy, ny - dy) ** 2)
            rad = min(nx, ny) * (0.04 + 0.08 * r[k, 2])
            d = torch.maximum(d, 0.5 * (1.0 - torch.tanh((dist - rad) / 2.0)))
        a = torch.tensor([0.8, 0.15, 0.05], **kw)[:, None, None, None]
        b = torch.tensor([0.15, 0.8, 0.05], **kw)[:, None, None, None]
        rho = a * d + b * (1.0 - d) + (0.01 if case["kind"] == "job" else 0.3) * noise
    elif start == "slab":       # 0.3 / 0.7 polymer solution against pure non-solvent
        left = torch.zeros(1, ny, nx, **kw)
        left[..., :nx // 2] = 1.0
        for c in (nx // 2 - 2, nx // 2 - 1, nx // 2, nx // 2 + 1, nx - 2, nx - 1, 0, 1):
            left[..., c] = 0.5 + 0.01 * (2.0 * rand(1, ny) - 1.0)
        rho = torch.stack([0.3 * left, 0.7 * left, 1.0 - left])
        del noise
    else:                       # "layers": the Sec. 4 sinusoid, polymer-poor to polymer-rich
        phi = [0.25] + [0.75 / (n - 1)] * (n - 1)
        wave = 0.1 * torch.sin(tp * x / nx + ph[0]) * (1.0 + 0.2 * torch.cos(tp * y / ny + ph[1]))
        rho = torch.tensor(phi, **kw)[:, None, None, None] + 0.2 * noise
        rho[0] += wave
        rho[1] -= wave
    amp = 0.01 if start in ("slab", "layers") else 0.03
    full = torch.zeros(nz, ny, nx, **kw)
    if case["kind"] == "cube":
        u = [0.01 + amp * torch.sin(tp * y / ny + ph[2]) + full, amp * torch.cos(tp * z / nz + ph[3]) + full,
             -0.005 + amp * torch.sin(tp * x / nx + ph[4]) + full]
    elif case["kind"] == "channel":
        prof = amp * torch.sin(math.pi * (y + 0.5) / ny)
        u = [prof + full, 0.2 * prof * torch.sin(tp * x / nx + ph[2]) + full]
    else:
        u = [0.01 + amp * torch.sin(tp * y / ny + ph[2]) + full, -0.005 + amp * torch.cos(tp * x / nx + ph[3]) + full]
    u = torch.stack(u)
    if case["kind"] != "cube":
        rho, u = rho.reshape(n, ny, nx), u.reshape(2, ny, nx)
    return rho.contiguous(), u.contiguous()


class _Instance:
    """One instance of a batch, with the attributes Batch reads."""

    def __init__(self, params, rho, u):
        self.__dict__.update(params)
        self.rho, self.u = rho, u


def _instances(case, seed, device):
    """(parameters, rho, u) of every instance of a batch or a sweep of lines."""
    rs = np.random.RandomState(seed % (1 << 31))
    shape = np.random.RandomState(4)    # the sizes belong to the case, not to the seed
    out = []
    for k in range(case["count"]):
        if case["kind"] == "batch":
            n = 2 + int(shape.randint(2))
            nx, ny = (int(shape.randint(case["lo"], case["hi"] + 1)) for _ in range(2))
            sub = dict(kind="plane", n=n, nx=nx, ny=ny, start="mixed", m0=1.0, kappa=0.01,
                       chi=2.0 * rs.uniform(0.9, 1.25), tau=rs.uniform(0.6, 1.5))
            rho, u = _fields(sub, seed + 1 + k, device)
            out.append((_params(sub, seed), rho, u))
        else:
            # a sweep along the Sec. 4 systems: interactions, relaxation times, compositions
            n, nx, m0 = case["n"], case["nx"], case["m0"]
            chi = np.zeros((n, n))
            chi[0, 1] = chi[1, 0] = rs.uniform(0.8, 0.9) if m0 > 1.0 else rs.uniform(1.9, 2.3)
            if n > 2:
                chi[0, 2] = chi[2, 0] = 0.5
                chi[1, 2] = chi[2, 1] = 0.2
            phi = np.full(n, 0.2)
            phi[0] = rs.uniform(0.2, 0.3) if m0 > 1.0 else rs.uniform(0.35, 0.45)
            phi[1] = 1.0 - phi[0] - phi[2:].sum()
            x = np.arange(nx)
            r = np.repeat(phi[:, None], nx, 1)
            w = 0.1 * np.sin(2.0 * math.pi * x / nx + rs.uniform(0, 6.28))
            r[0] += w
            r[1] -= w
            m = np.ones(n)
            m[0] = m0
            p = dict(ncomp=n, nx=nx, ny=1, nz=1, tau=1.0 / rs.uniform(0.7, 0.95), chi=chi, m=m,
                     theta=1.0 / 3.0, kappa=0.0, force=(0.0, 0.0), forcing_velocity=1,
                     force_form=case["gd"], lattice="d1q3", walls=0)
            uu = np.zeros((2, 1, nx))
            uu[0] = 0.01 + 0.01 * np.cos(2.0 * math.pi * x / nx)
            out.append((p, torch.from_numpy(r.reshape(n, 1, nx)), torch.from_numpy(uu)))
    return out


def prepare(case, seed):
    kind, prec = case["kind"], case["precision"]
    snap = torch.float64 if prec == "fp64" else torch.float32
    if kind in ("batch", "lines"):
        items = [_Instance(p, r.cpu().numpy(), u.cpu().numpy())
                 for p, r, u in _instances(case, seed, "cuda")]
        b = mclb.Batch(items, precision=prec)
        b.init_all()
        return dict(case=case, batch=b, count=len(items), np=np.float64 if prec == "fp64" else np.float32)
    p = _params(case, seed)
    rho, u = _fields(case, seed, "cuda")
    if p["lattice"] == "d2q9":
        p["nz"] = 1
    sim = mclb.Simulation(precision=prec, **p)
    if kind == "job":
        return dict(case=case, sim=sim, rho=rho.cpu().numpy(), u=u.cpu().numpy(),
                    np=np.float64 if prec == "fp64" else np.float32)
    sim.init_fields_device(rho, u)
    torch.cuda.synchronize()
    mu = None if case.get("start") == "slab" else torch.empty_like(rho)
    return dict(case=case, sim=sim, rho=rho, u=u, mu=mu, snap=snap)


def run(state):
    case = state["case"]
    if "batch" in state:
        b = state["batch"]
        b.step(case["steps"])
        got = [b.moments(k) for k in range(state["count"])]
        return [np.concatenate([m[f].ravel() for m in got]).astype(state["np"], copy=False) for f in ("rho", "U")]
    sim = state["sim"]
    if case["kind"] == "job":
        sim.init_fields(state["rho"], state["u"])
        sim.step(case["steps"])
        m = sim.moments()
        sums = sim.conservation()
        fit = sim.fit_equilibrium(2)
        return [m[f].astype(state["np"], copy=False) for f in ("rho", "U", "mu")] + \
               [sums["mass"].astype(state["np"]), sums["mom"].astype(state["np"]), fit.astype(np.float32)]
    sim.step(case["steps"])
    sim.moments_device(rho=state["rho"], U=state["u"], mu=state["mu"])
    return [f.to(state["snap"]) for f in (state["rho"], state["u"], state["mu"]) if f is not None]


def work(case):
    """Bytes: every timestep reads and writes each stored value once (a lattice is advanced
    step by step; D1Q3 lines cross memory once per pass, since a line is held on chip), and
    the fields are written once.  Flops: the additions and multiplications of the equations
    per component (moments, stencils, potential, forcing and collision over the velocities)
    and per site (u, the equilibrium weights, one logarithm)."""
    v, r = PRECISION_BYTES[case["precision"]]
    kind = case["kind"]
    steps = case["steps"]
    if kind == "batch":
        shape, site_n, sites = np.random.RandomState(4), 0, 0
        flops = 0
        for _ in range(case["count"]):
            n = 2 + int(shape.randint(2))
            s = int(shape.randint(case["lo"], case["hi"] + 1)) * int(shape.randint(case["lo"], case["hi"] + 1))
            site_n += n * s
            sites += s
            flops += s * (n * (135 + 2 * n) + 70)
        return {"bytes": 2.0 * site_n * (9 * v + r) * steps + 8.0 * (site_n + 2 * sites),
                "flops": float(flops) * steps}
    n = case["n"]
    if kind == "lines":
        s = case["count"] * case["nx"]
        return {"bytes": 2.0 * n * s * 3 * v + 8.0 * s * (n + 2), "flops": float(s) * (n * (45 + 2 * n) + 25) * steps}
    s = case["nx"] * case["ny"] * case.get("nz", 1)
    out = 8.0 * s * ((2 if case.get("start") != "slab" else 1) * n + (3 if kind == "cube" else 2))
    if kind == "cube":
        return {"bytes": 2.0 * n * s * 19 * v * steps + out, "flops": float(s) * (n * (300 + 2 * n) + 130) * steps}
    return {"bytes": 2.0 * n * s * (9 * v + r) * steps + out, "flops": float(s) * (n * (135 + 2 * n) + 70) * steps}


# ---------------------------------------------------------------- the method in 64 bits

_C1 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0)]
_C2 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
_C3 = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1) if abs(x) + abs(y) + abs(z) < 3]


class _Exact:
    """Pre-collision populations f (N, Q, z, y, x), advanced by the equations in FP64."""

    def __init__(self, p, rho, u):
        lat = p["lattice"]
        self.p, self.dev = p, rho.device
        self.c = {"d1q3": _C1, "d2q9": _C2, "d3q19": _C3}[lat]
        wt = {"d1q3": {0: 2 / 3, 1: 1 / 6}, "d2q9": {0: 4 / 9, 1: 1 / 9, 2: 1 / 36},
              "d3q19": {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}}[lat]
        self.w = [wt[sum(abs(v) for v in c)] for c in self.c]
        n, nz, ny, nx = p["ncomp"], p["nz"], p["ny"], p["nx"]
        rho = rho.reshape(n, nz, ny, nx)
        u = u.reshape(-1, nz, ny, nx)
        self.ud = u.shape[0]
        self.dims = 1 if lat == "d1q3" else self.ud
        uu = sum(u[d] ** 2 for d in range(self.dims))
        self.f = [[self.w[i] * rho[s] * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
                   for i, cu in enumerate(self._dots(u))] for s in range(n)]

    def _dots(self, a):
        return [sum((a[d] * c[d] for d in range(self.dims) if c[d]), torch.zeros_like(a[0])) for c in self.c]

    def _at(self, g, c):
        """g(x + c): periodic, or the mirrored rows beyond a wall."""
        if c[1] and self.p["walls"]:
            g = torch.cat([g[:, 1:], g[:, -1:]], 1) if c[1] > 0 else torch.cat([g[:, :1], g[:, :-1]], 1)
            c = (c[0], 0, c[2])
        return torch.roll(g, (-c[2], -c[1], -c[0]), (0, 1, 2)) if any(c) else g

    def _grad(self, g):
        out = [torch.zeros_like(g) for _ in range(self.dims)]
        for w, c in zip(self.w, self.c):
            if any(c):
                v = 3 * w * self._at(g, c)
                for d in range(self.dims):
                    if c[d]:
                        out[d] += c[d] * v
        return out

    def _lap(self, g):
        if self.p["kappa"] == 0.0:
            return torch.zeros_like(g)
        return 6 * sum(w * (self._at(g, c) - g) for w, c in zip(self.w, self.c) if any(c))

    def _site(self):
        """Densities, momenta, u and the accelerations of the current state."""
        p, n = self.p, self.p["ncomp"]
        r = [sum(f) for f in self.f]
        j = [[sum(c[d] * f[i] for i, c in enumerate(self.c) if c[d]) for d in range(self.dims)] for f in self.f]
        rho = sum(r)
        u = [sum(j[s][d] for s in range(n)) / rho for d in range(self.dims)]
        k = 1.0 - 1.0 / (2.0 * p["tau"])
        bulk, mu = self._mu_bulk(r, rho)
        lap = [self._lap(r[s]) for s in range(n)]
        a = []
        for s in range(n):
            th = p["theta"] / p["m"][s]
            nu = bulk[s] - th * torch.log(rho) - p["kappa"] * lap[s]
            if th - 1.0 / 3.0 != 0.0:
                nu = nu + (th - 1.0 / 3.0) * torch.log(torch.maximum(r[s], 1e-12 * rho))
            a.append([-k * g + p["force"][d] for d, g in enumerate(self._grad(nu))])
        if p["force_form"]:
            gr = self._grad(rho)
            for d in range(self.dims):
                tot = sum(r[s] * (a[s][d] - p["force"][d]) for s in range(n))
                sh = (k / 3.0 * gr[d] - tot) / rho
                for s in range(n):
                    a[s][d] = a[s][d] + sh
        return r, j, rho, u, a, [mu[s] - p["kappa"] * lap[s] for s in range(n)]

    def _mu_bulk(self, r, rho):
        """(theta [1/m - 1 - sum phi/m + chi phi - phi chi phi / 2], that + theta ln(phi)/m)."""
        p, n = self.p, self.p["ncomp"]
        phi = [r[s] / rho for s in range(n)]
        sm = sum(phi[s] / p["m"][s] for s in range(n))
        cp = [sum((p["chi"][s, t] * phi[t] for t in range(n) if t != s), torch.zeros_like(rho)) for s in range(n)]
        quad = 0.5 * sum(phi[s] * cp[s] for s in range(n))
        bulk = [p["theta"] * (1.0 / p["m"][s] - 1.0 - sm + cp[s] - quad) for s in range(n)]
        mu = [bulk[s] + p["theta"] / p["m"][s] * torch.log(torch.clamp(phi[s], min=1e-12)) for s in range(n)]
        return bulk, mu

    def step(self):
        p, om = self.p, 1.0 / self.p["tau"]
        r, j, rho, u, a, _ = self._site()
        uu = sum(v * v for v in u)
        cu = self._dots(u)
        for s in range(p["ncomp"]):
            js = [r[s] * v for v in u] if p["forcing_velocity"] else j[s]
            ca, cj = self._dots(a[s]), self._dots(js)
            aj = sum(x * y for x, y in zip(a[s], js))
            post = []
            for i, w in enumerate(self.w):
                fe = w * r[s] * (1 + 3 * cu[i] + 4.5 * cu[i] * cu[i] - 1.5 * uu)
                F = w * (3 * r[s] * ca[i] + 9 * ca[i] * cj[i] - 3 * aj)
                post.append(self.f[s][i] + om * (fe - self.f[s][i]) + F)
            for i, c in enumerate(self.c):
                g = torch.roll(post[i], (c[2], c[1], c[0]), (0, 1, 2)) if any(c) else post[i]
                if c[1] and p["walls"]:     # what would cross a wall returns reversed to its site
                    o = self.c.index((-c[0], -c[1], -c[2]))
                    row = 0 if c[1] > 0 else -1
                    g[:, row] = post[o][:, row]
                self.f[s][i] = g

    def moments(self):
        r, j, rho, u, a, mu = self._site()
        n = self.p["ncomp"]
        U = [u[d] + 0.5 * sum(r[s] * a[s][d] for s in range(n)) / rho for d in range(self.dims)]
        U += [torch.zeros_like(rho)] * (self.ud - self.dims)
        return torch.stack(r), torch.stack(U), torch.stack(mu)


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "lines":
        return _exact_lines(case, seed, dev)
    if kind == "batch":
        rho, U = [], []
        for p, r, u in _instances(case, seed, dev):
            e = _Exact(p, r, u)
            for _ in range(case["steps"]):
                e.step()
            m = e.moments()
            rho.append(m[0].ravel().cpu())
            U.append(m[1].ravel().cpu())
        return [torch.cat(rho), torch.cat(U)]
    p = _params(case, seed)
    rho, u = _fields(case, seed, dev)
    shape, ushape = rho.shape, u.shape
    e = _Exact(p, rho, u)
    del rho, u
    for _ in range(case["steps"]):
        e.step()
    r, U, mu = e.moments()
    out = [r.reshape(shape), U.reshape(ushape), None if case.get("start") == "slab" else mu.reshape(shape)]
    if kind == "job":
        j = e._site()[1]
        out += [r.reshape(case["n"], -1).sum(1), torch.stack([sum(j[s][d] for s in range(case["n"])).sum() for d in range(2)]), None]
    return out if kind == "job" else out[:2 if case.get("start") == "slab" else 3]


def _exact_lines(case, seed, dev):
    """Every line of a sweep at once: the lines are rows, which a D1Q3 step does not couple, and
    what differs from line to line (tau, chi) is a column of values."""
    items = _instances(case, seed, dev)
    n = case["n"]
    p = dict(items[0][0])
    p["ny"] = len(items)

    def column(values):
        return torch.tensor(values, device=dev, dtype=torch.float64)[None, :, None]

    p["tau"] = column([q[0]["tau"] for q in items])
    p["chi"] = {(a, b): column([q[0]["chi"][a, b] for q in items]) for a in range(n) for b in range(n)}
    e = _Exact(p, torch.cat([q[1] for q in items], 1).to(dev), torch.cat([q[2] for q in items], 1).to(dev))
    for _ in range(case["steps"]):
        e.step()
    r, U, _ = e.moments()
    r, U = r[:, 0], U[:, 0]                        # (n, lines, nx), (2, lines, nx)
    return [r.permute(1, 0, 2).reshape(-1), U.permute(1, 0, 2).reshape(-1)]
