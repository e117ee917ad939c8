"""Workloads of the library, each one pass through its public entry points.

Kinds of case (the "kind" of a case's dict):
  box       a fluctuating run as the paper's: a periodic box in thermal equilibrium advances
            `steps` steps and its populations are read into device memory
  hydro     a deterministic run (kT = 0): initial density and velocity fields, `steps` steps,
            then density, velocity and stress in FP64 device memory
  coupled   a step inside another solver's loop: its float32 populations in, `steps` steps,
            populations and global statistics out, everything on the device
  snapshot  one sample of the equilibrium statistics: global statistics, the 27 mode sums and
            the structure factors of the ten hydrodynamic fields
  ensemble  many small boxes of their own tau, kT and seed advanced together from rest, then
            the populations of each
  slabs     one box split along z over several handles that exchange their faces every step

Inputs are thermal: f_i = w_i rho0 plus independent normals of variance 3 kT w_i rho0, whose 27
modes have the fluctuation-dissipation variances. `exact` restates the model in FP64 torch
(arXiv 2507.08820, Eqs. 3-12 and 21-26, with the library's documented noise generator).
"""
import math

import numpy as np
import torch

from paper_2507_08820_gb300 import rflbm as R

_STORAGE = {"f32": R.RFLBM_STORE_F32, "f16": R.RFLBM_STORE_F16, "bf16": R.RFLBM_STORE_BF16}
_ELEM = {"f32": 4, "f16": 2, "bf16": 2}
_PATTERN = {"pingpong": R.RFLBM_PATTERN_PINGPONG, "aa": R.RFLBM_PATTERN_AA}
_MODEL = {"reg": R.RFLBM_MODEL_REG, "bgk": R.RFLBM_MODEL_BGK}


def _box(name, nx, ny, nz, steps, storage="f32", pattern="pingpong", model="reg", tau=0.8, kT=1e-4):
    return dict(name=name, kind="box", nx=nx, ny=ny, nz=nz, steps=steps, storage=storage, pattern=pattern,
                model=model, tau=tau, kT=kT)


def listed():
    return [
        # the smallest configuration of the parity tests (32^3 x 100 steps): launches and latency
        _box("box_32", 32, 32, 32, 100),
        # the benchmark's configuration: the fluctuating step at 128^3 in float32
        _box("box_128", 128, 128, 128, 20),
        # an edge that no power of two divides, rows of whole 16-byte units
        _box("box_100", 100, 100, 100, 20),
        # an uneven box whose rows are no whole number of 16-byte units
        _box("box_150x110x70", 150, 110, 70, 20),
        # 16-bit population storage (the mixed-precision configuration)
        _box("box_256_f16", 256, 256, 256, 10, storage="f16"),
        # the in-place pattern with 16-bit storage: boxes chosen for their size in memory
        _box("aa_512x448x384_f16", 512, 448, 384, 4, storage="f16", pattern="aa"),
        # the model that the paper compares against, in its stable range
        _box("bgk_128", 128, 128, 128, 20, model="bgk", tau=0.55),
        # a Taylor-Green vortex without noise, measured by its velocity and stress fields
        dict(name="hydro_192", kind="hydro", nx=192, ny=192, nz=192, steps=20, storage="f32", pattern="pingpong", tau=0.6),
        # one step per exchange with another solver that keeps its own populations
        dict(name="coupled_96x80x72", kind="coupled", nx=96, ny=80, nz=72, steps=1, storage="f32", pattern="pingpong",
             tau=0.7, kT=1e-4),
        # one sample of the equilibration ratios and spectra (Table III, Figs. 1-2)
        dict(name="snapshot_128", kind="snapshot", nx=128, ny=128, nz=128, storage="f32", tau=0.51, kT=1 / 3000),
        # a parameter scan over small boxes
        dict(name="ensemble_16", kind="ensemble", replicas=16, edges="16,24,32", steps=400, storage="f32"),
        # the paper's linear domain decomposition, its slabs on one device
        dict(name="slabs_2x128x128x64", kind="slabs", nx=128, ny=128, nz=128, slabs=2, steps=10, storage="f32",
             pattern="pingpong", tau=0.8, kT=1e-4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    case = _draw(rng)
    most = max(work(c)["bytes"] for c in listed())
    while work(case)["bytes"] > most and case.get("steps", 1) > 1:
        case["steps"] = max(1, int(0.9 * case["steps"] * most / work(case)["bytes"]))
    return case


def _draw(rng):
    kind = rng.choice(["box", "box", "box", "box", "hydro", "coupled", "snapshot", "ensemble", "slabs"])
    # edges over their logarithm, half of them whole multiples of 8
    edge = lambda lo, hi: (lambda e: e if rng.random() < 0.5 else max(lo, e // 8 * 8))(_log(rng, lo, hi))  # noqa: E731
    storage = rng.choice(["f32", "f32", "f16", "bf16"])
    pattern = rng.choice(["pingpong", "pingpong", "aa"])
    tau, kT = round(rng.uniform(0.55, 1.5), 3), float("%.3g" % 10 ** rng.uniform(-5, -3))
    if kind == "box":
        return dict(kind=kind, nx=edge(16, 384), ny=edge(16, 256), nz=edge(16, 256), steps=_log(rng, 4, 100),
                    storage=storage, pattern=pattern, model=rng.choice(["reg", "reg", "bgk"]), tau=tau, kT=kT)
    if kind == "hydro":
        e = edge(24, 256)
        return dict(kind=kind, nx=e, ny=e, nz=edge(8, 256), steps=_log(rng, 4, 40), storage="f32", pattern=pattern, tau=tau)
    if kind == "coupled":
        return dict(kind=kind, nx=edge(16, 192), ny=edge(16, 192), nz=edge(16, 192), steps=rng.randint(1, 4),
                    storage=storage, pattern=pattern, tau=tau, kT=kT)
    if kind == "snapshot":
        return dict(kind=kind, nx=edge(32, 192), ny=edge(32, 192), nz=edge(32, 192), storage=storage, tau=tau, kT=kT)
    if kind == "ensemble":
        edges = ",".join(str(rng.choice([16, 20, 24, 32, 33, 40, 48])) for _ in range(rng.randint(1, 3)))
        return dict(kind=kind, replicas=rng.randint(4, 24), edges=edges, steps=_log(rng, 100, 400), storage=storage)
    return dict(kind=kind, nx=edge(32, 160), ny=edge(32, 160), nz=edge(32, 160), slabs=rng.randint(1, 3),
                steps=rng.randint(2, 12), storage=storage, pattern=pattern, tau=tau, kT=kT)


# ------------------------------------------------------------------ inputs
def _weights():
    w1 = {0: 2.0 / 3.0, 1: 1.0 / 6.0, -1: 1.0 / 6.0}
    return [w1[x] * w1[y] * w1[z] for x, y, z in _C]


def _thermal(n, kT, seed):
    """float32 populations (27, n) of a box in thermal equilibrium around the rest state."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.empty((27, n), dtype=torch.float32, device="cuda")
    for i, w in enumerate(_weights()):
        f[i].normal_(generator=g).mul_(math.sqrt(3.0 * kT * w)).add_(w)
    return f


def _vortex(case, seed):
    """FP64 density (n) and velocity (3, n) of a Taylor-Green vortex with a phase and an
    amplitude of the seed's."""
    rng = np.random.default_rng(seed)
    u0, px, py = rng.uniform(0.01, 0.03), *rng.uniform(0, 2 * np.pi, 2)
    s = torch.arange(_sites(case), device="cuda")
    k = 2 * math.pi / case["nx"]
    x = k * (s % case["nx"]).double() + px
    y = k * ((s // case["nx"]) % case["ny"]).double() + py
    u = torch.stack([-u0 * torch.cos(x) * torch.sin(y), u0 * torch.sin(x) * torch.cos(y), torch.zeros_like(x)])
    return 1.0 - 0.75 * u0 * u0 * (torch.cos(2 * x) + torch.cos(2 * y)), u


def _replicas(case, seed):
    rng = np.random.default_rng(seed)
    edges = [int(e) for e in case["edges"].split(",")]
    return [dict(nx=edges[i % len(edges)], ny=edges[i % len(edges)], nz=edges[i % len(edges)],
                 tau=float(rng.uniform(0.55, 1.2)), kT=float(10 ** rng.uniform(-5, -3)), seed=int(rng.integers(1, 1 << 40)))
            for i in range(case["replicas"])]


def _slab_rows(case):
    k, nz = case["slabs"], case["nz"]
    cuts = [nz * i // k for i in range(k + 1)]
    return [(a, b - a) for a, b in zip(cuts[:-1], cuts[1:])]


def _sites(case):
    return case["nx"] * case["ny"] * case["nz"]


def _handle(case, seed, **more):
    return R.Box(case["nx"], case["ny"], more.pop("nz", case["nz"]), tau=case["tau"], kT=case.get("kT", 0.0), seed=seed + 1,
                 storage=_STORAGE[case["storage"]], pattern=_PATTERN[case.get("pattern", "pingpong")],
                 model=_MODEL[case.get("model", "reg")], **more)


class _Ensemble:
    """An ensemble's handle, released with its state."""

    def __init__(self, case, seed):
        self.reps = _replicas(case, seed)
        self.b = R.rflbm_batch_create(self.reps, storage=_STORAGE[case["storage"]])
        R.rflbm_batch_init_rest(self.b)
        R.rflbm_batch_prepare(self.b, case["steps"])
        self.f = [np.full((27, r["nx"] * r["ny"] * r["nz"]), 0.0) for r in self.reps]

    def __del__(self):
        R.rflbm_batch_destroy(self.b)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        return dict(case=case, batch=_Ensemble(case, seed))
    n, dev = _sites(case), "cuda"
    if kind == "slabs":
        f = _thermal(n, case["kT"], seed).view(27, case["nz"], case["ny"] * case["nx"])
        boxes, outs = [], []
        for z0, nz in _slab_rows(case):
            box = _handle(case, seed, nz=nz, z0=z0, nz_global=case["nz"])
            mine = f[:, z0:z0 + nz].reshape(27, -1).contiguous()
            R.rflbm_set_populations_f32(box.h, mine)
            boxes.append(box)
            outs.append(mine)
        torch.cuda.synchronize()
        return dict(case=case, boxes=boxes, outs=outs)
    box = _handle(case, seed)
    if kind == "hydro":
        rho, u = _vortex(case, seed)
        out = [torch.empty(s, dtype=torch.float64, device=dev) for s in ((n,), (3, n), (6, n))]
        return dict(case=case, box=box, rho=rho, u=u, out=out)
    f = _thermal(n, case["kT"], seed)
    if kind == "coupled":
        return dict(case=case, box=box, f=f, out=torch.empty_like(f))
    R.rflbm_set_populations_f32(box.h, f)
    torch.cuda.synchronize()
    return dict(case=case, box=box, out=f if kind == "box" else None)


# ------------------------------------------------------------------ one pass
def _stats(st):
    return np.array([st.mass, *st.momentum, st.max_speed]), int(st.nonfinite)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "box":
        h = state["box"].h
        R.rflbm_step(h, case["steps"])
        R.rflbm_get_populations_f32(h, state["out"])
        return state["out"]
    if kind == "hydro":
        h = state["box"].h
        R.rflbm_init_field(h, state["rho"], state["u"])
        R.rflbm_step(h, case["steps"])
        R.rflbm_moments(h, *state["out"])
        return state["out"]
    if kind == "coupled":
        h = state["box"].h
        R.rflbm_set_populations_f32(h, state["f"])
        R.rflbm_step(h, case["steps"])
        R.rflbm_get_populations_f32(h, state["out"])
        return [state["out"], *_stats(R.rflbm_stats(h)[0])]
    if kind == "snapshot":
        h = state["box"].h
        stats = _stats(R.rflbm_stats(h)[0])
        sums = R.rflbm_mode_sums(h)
        spectra = [R.rflbm_structure_factor(h, field) for field in R.FIELDS]
        return [*stats, *sums, np.array([s for s, _ in spectra]), np.array([c for _, c in spectra])]
    if kind == "ensemble":
        e = state["batch"]
        R.rflbm_batch_run(e.b, case["steps"])
        for r, f in enumerate(e.f):
            R.rflbm_batch_get_populations(e.b, r, f)
        return e.f
    handles = [b.h for b in state["boxes"]]
    for _ in range(case["steps"]):
        for h in handles:
            R.rflbm_step(h, 1)
        R.rflbm_slab_exchange(handles)
    for h, out in zip(handles, state["outs"]):
        R.rflbm_get_populations_f32(h, out)
    return state["outs"]


def work(case):
    """Populations read and written once a step, inputs read and outputs written once; the
    floating-point operations of the factorised transforms and of the 24 normals of a site."""
    kind = case["kind"]
    e = _ELEM[case["storage"]]
    if kind == "ensemble":
        edges = [int(x) for x in case["edges"].split(",")]
        n = sum(edges[i % len(edges)] ** 3 for i in range(case["replicas"]))
        return dict(bytes=n * (54 * e * case["steps"] + 27 * (e + 8)), flops=n * case["steps"] * 500)
    n = _sites(case)
    if kind == "snapshot":  # the state once, and ten fields with their spectra (FP64, 5/2 n log2 n)
        return dict(bytes=n * 27 * e, flops=10 * (n * 30 + 2.5 * n * math.log2(n)) + n * 200)
    steps = case["steps"]
    if kind == "hydro":
        return dict(bytes=n * (54 * e * steps + 27 * 2 * e + 4 * 8 + 10 * 8), flops=n * (280 * steps + 300))
    if kind == "coupled":
        return dict(bytes=n * (54 * e * steps + 27 * 2 * (e + 4)), flops=n * 500 * steps)
    return dict(bytes=n * (54 * e * steps + 27 * (e + 4)), flops=n * 500 * steps)


# ------------------------------------------------------------------ the model in FP64
# velocities in the order of include/rflbm.h, and the Hermite exponents of the 27 modes (Table II)
_C = ([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
      + [(a, b, 0) for a in (1, -1) for b in (1, -1)] + [(a, 0, b) for a in (1, -1) for b in (1, -1)]
      + [(0, a, b) for a in (1, -1) for b in (1, -1)]
      + [(a, b, c) for a in (1, -1) for b in (1, -1) for c in (1, -1)])
_P = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1),
      (2, 1, 0), (2, 0, 1), (1, 2, 0), (1, 0, 2), (0, 1, 2), (0, 2, 1), (1, 1, 1), (2, 2, 0), (2, 0, 2), (0, 2, 2),
      (1, 1, 2), (1, 2, 1), (2, 1, 1), (2, 1, 2), (2, 2, 1), (1, 2, 2), (2, 2, 2)]
_MASK = 0xFFFFFFFF
_CHUNK = 1 << 23  # sites collided at once


def _philox(site, step, call, key0, key1):
    """The four words (int64) of Philox4x32-10 at counter (site, step, call, 0)."""
    def mul(m, c):
        p0, p1 = m * (c & 0xFFFF), m * (c >> 16)
        low = p0 + ((p1 & 0xFFFF) << 16)
        return (p1 >> 16) + (low >> 32), low & _MASK
    c = [site, torch.full_like(site, step), torch.full_like(site, call), torch.zeros_like(site)]
    for r in range(10):
        hi0, lo0 = mul(0xD2511F53, c[0])
        hi1, lo1 = mul(0xCD9E8D57, c[2])
        c = [hi1 ^ c[1] ^ ((key0 + r * 0x9E3779B9) & _MASK), lo1, hi0 ^ c[3] ^ ((key1 + r * 0xBB67AE85) & _MASK), lo0]
    return c


def _normals(site, step, key0, key1):
    """The 24 normals of each site: Box-Muller on word pairs (0, 1) and (2, 3) of calls 0..5."""
    out = []
    for call in range(6):
        u = [(w.double() + 0.5) * 2.0 ** -32 for w in _philox(site, step, call, key0, key1)]
        for a, b in ((u[0], u[1]), (u[2], u[3])):
            r = torch.sqrt(-2.0 * torch.log(a))
            out += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
    return out


class _Model:
    """One or more boxes as flat FP64 populations (27, n): tau, kT and key per site or for all."""

    def __init__(self, f, tau, kT, key, bgk=False, site=None):
        h = lambda p, c: (1.0, c, c * c - 1.0 / 3.0)[p]  # noqa: E731
        e = [[h(p, x) * h(q, y) * h(r, z) for x, y, z in _C] for p, q, r in _P]
        beta = (1.0, 1.0 / 3.0, 2.0 / 9.0)
        self.b = [beta[p] * beta[q] * beta[r] for p, q, r in _P]
        self.e = torch.tensor(e, dtype=torch.float64, device="cuda")
        w = torch.tensor(_weights(), dtype=torch.float64, device="cuda")
        self.back = (self.e / torch.tensor(self.b, dtype=torch.float64, device="cuda")[:, None] * w).T.contiguous()
        self.f, self.tau, self.kT, self.key, self.bgk, self.site, self.t = f, tau, kT, key, bgk, site, 0

    def collide(self):
        n = self.f.shape[1]
        at = lambda v, s: v[s] if torch.is_tensor(v) else v  # noqa: E731
        for a in range(0, n, _CHUNK):
            s = slice(a, min(n, a + _CHUNK))
            f = self.f[:, s]
            m = self.e[:27 if self.bgk else 10] @ f
            rho = m[0]
            u = [m[k] / rho for k in (1, 2, 3)]
            om, kT = 1.0 / at(self.tau, s), at(self.kT, s)
            noisy = torch.is_tensor(kT) or kT > 0
            if noisy:
                site = self.site[s] if self.site is not None else torch.arange(s.start, s.stop, device="cuda")
                r = _normals(site, self.t, at(self.key[0], s), at(self.key[1], s))
            new = torch.empty((27, rho.numel()), dtype=torch.float64, device="cuda")
            new[:4] = m[:4]
            for k in range(4, 27):
                p, q, o = _P[k]
                eq = rho * u[0] ** p * u[1] ** q * u[2] ** o
                rate = om if self.bgk or k < 10 else 1.0
                new[k] = rate * eq + (1.0 - rate) * m[k] if self.bgk or k < 10 else eq
                if noisy:
                    new[k] += torch.sqrt(3.0 * self.b[k] * rho * kT * rate * (2.0 - rate)) * r[k - 4]
            self.f[:, s] = self.back @ new
        self.t += 1

    def step(self, shape):
        """shape: (nz, ny, nx) of a box, or the source sites (27, n) of the streaming."""
        self.collide()
        if torch.is_tensor(shape):
            for i in range(27):
                self.f[i] = self.f[i][shape[i]]
            return
        for i, (x, y, z) in enumerate(_C):
            if i:
                self.f[i] = torch.roll(self.f[i].view(shape), (z, y, x), (0, 1, 2)).reshape(-1)

    def fields(self):
        m = self.e[:10] @ self.f
        return m[0], m[1:4] / m[0], m[4:10]


def _exact_stats(model):
    rho, u, _ = model.fields()
    j = (u * rho).sum(1)
    return torch.stack([rho.sum(), *j, u.square().sum(0).sqrt().max()]).cpu().numpy(), None


def _exact_snapshot(case, model):
    shape = (case["nz"], case["ny"], case["nx"])
    n, L = _sites(case), max(shape)
    m = model.e @ model.f
    m[0] -= 1.0
    k2 = sum((torch.fft.fftfreq(e, dtype=torch.float64, device="cuda") ** 2).view(v)
             for e, v in zip(shape, ((-1, 1, 1), (1, -1, 1), (1, 1, -1))))
    shell = torch.round(L * torch.sqrt(k2)).long().reshape(-1)
    ns = int(round(L * math.sqrt(3.0) / 2.0)) + 1
    s = np.array([torch.zeros(ns, dtype=torch.float64, device="cuda").index_add_(
        0, shell, (torch.fft.fftn(m[k].view(shape)).abs().square() / n).reshape(-1)).cpu().numpy() for k in range(10)])
    counts = np.tile(torch.bincount(shell, minlength=ns).double().cpu().numpy(), (10, 1))
    return [*_exact_stats(model), m.sum(1).cpu().numpy(), m.square().sum(1).cpu().numpy(), s, counts]


def _exact_ensemble(case, seed):
    reps = _replicas(case, seed)
    sizes = [r["nx"] ** 3 for r in reps]
    per = lambda key, dtype: torch.cat([torch.full((n,), key(r), dtype=dtype, device="cuda") for r, n in zip(reps, sizes)])  # noqa: E731
    source, base = [], 0
    for r, n in zip(reps, sizes):
        grid = torch.arange(n, device="cuda").view(r["nz"], r["ny"], r["nx"])
        source.append(torch.stack([torch.roll(grid, (z, y, x), (0, 1, 2)).reshape(-1) for x, y, z in _C]) + base)
        base += n
    f = torch.tensor(_weights(), dtype=torch.float64, device="cuda")[:, None].repeat(1, base)
    model = _Model(f, per(lambda r: r["tau"], torch.float64), per(lambda r: r["kT"], torch.float64),
                   (per(lambda r: r["seed"] & _MASK, torch.int64), per(lambda r: r["seed"] >> 32, torch.int64)),
                   site=torch.cat([torch.arange(n, device="cuda") for n in sizes]))
    source = torch.cat(source, 1)
    for _ in range(case["steps"]):
        model.step(source)
    return [x.cpu().numpy() for x in torch.split(model.f, sizes, 1)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        return _exact_ensemble(case, seed)
    shape = (case["nz"], case["ny"], case["nx"])
    if kind == "hydro":
        rho, u = _vortex(case, seed)
        psi = lambda c, v: 2.0 / 3.0 - v * v if c == 0 else 0.5 * (1.0 / 3.0 + c * v + v * v)  # noqa: E731
        f = torch.stack([rho * psi(x, u[0]) * psi(y, u[1]) * psi(z, u[2]) for x, y, z in _C])
    else:
        f = _thermal(_sites(case), case["kT"], seed).double()
    key = seed + 1
    model = _Model(f, case["tau"], case.get("kT", 0.0), (key & _MASK, key >> 32), bgk=case.get("model") == "bgk")
    if kind == "snapshot":
        return _exact_snapshot(case, model)
    for _ in range(case["steps"]):
        model.step(shape)
    if kind == "hydro":
        return list(model.fields())
    if kind == "coupled":
        return [model.f, *_exact_stats(model)]
    if kind == "slabs":
        rows = case["nx"] * case["ny"]
        return [model.f[:, z0 * rows:(z0 + nz) * rows] for z0, nz in _slab_rows(case)]
    return model.f
