"""The work this framework is used for, as cases that can be timed and compared.

A case is a plain dict. Its "kind" says which program it stands for:

  run       one lattice advanced by some steps with a diagnostics record: the time loop of
            every simulation here (small boxes to 512^3, cubes and ragged boxes, all stencil
            pairs, forcings and storage types)
  batch     a parameter sweep: many lattices of different sizes, pairs and forcings advanced
            together, then every instance's record and fields
  slab      one periodic lattice cut into z-slabs that exchange halos around every odd step
  restart   host fields in, a few steps, host fields out: starting from and saving snapshots
  analysis  the records and fields of a state on the GPU, for spectra and budgets

Physics is the stratified Taylor-Green vortex of the repository's benchmark (U0 = 0.04, Pr = 1)
with seeded noise on the velocity.
"""
import math

import torch

from paper_2605_14505_gb300 import halo, lbm

U0 = 0.04
NOISE = 1e-3
PAIRS = {"27x19": (27, 19), "19x7": (19, 7), "27x27": (27, 27), "19x19": (19, 19), "19x15": (19, 15),
         "15x7": (15, 7), "7x27": (7, 27)}
BYTES = {"fp32": 4, "fp16": 2, "bf16": 2}
TYPES = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}


def _run(name, nx, ny, nz, pair, forcing, storage, steps, record, Re=400.0, Fr=0.1):
    c = {"kind": "run", "nx": nx, "ny": ny, "nz": nz, "pair": pair, "forcing": forcing, "storage": storage,
         "steps": steps, "record": record, "Re": Re, "Fr": Fr}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small box whose record is read at every step (a coupled or monitored run): launch latency
        _run("monitor_32", 32, 32, 32, "19x7", "sc", "fp32", 1, "fused", 100.0, 0.5),
        # the smallest whole simulation of the benchmark list: 200 steps, then its record
        _run("box_32", 32, 32, 32, "27x19", "guo", "fp32", 200, "after", 100.0, 0.5),
        # the coarse grid of the resolution study with the cheap stencil pair
        _run("tgv_64", 64, 64, 64, "19x7", "guo", "fp32", 100, "fused", 200.0, 0.5),
        # the 128^3 series: a record every 50 steps
        _run("tgv_128", 128, 128, 128, "27x19", "sc", "fp32", 50, "fused", 400.0, 0.1),
        # the headline run, FP32 storage: a record every 100 steps
        _run("tgv_256_fp32", 256, 256, 256, "27x19", "sc", "fp32", 100, "fused", 800.0, 0.1),
        # the same with 16-bit deviation storage
        _run("tgv_256_fp16", 256, 256, 256, "27x19", "sc", "fp16", 100, "after", 800.0, 0.1),
        # the largest lattice: 25 GB of populations
        _run("tgv_512", 512, 512, 512, "27x19", "sc", "fp32", 20, "fused", 1600.0, 0.1),
        # a box that is no cube and has odd sides, 16-bit storage
        _run("ragged", 225, 150, 75, "27x19", "edm", "fp16", 50, "after", 400.0, 0.2),
        # the sweep over size, Froude number, forcing and pair: 64 instances, 20.6 million nodes
        {"name": "sweep_64", "kind": "batch", "mode": "instances", "sizes": "32,48,64,96", "frs": "1,0.5,0.2,0.1",
         "forcings": "guo,sc", "pairs": "19x7,27x19", "Re": 200.0, "steps": 100},
        # a z-decomposed lattice: halos travel around every odd step
        {"name": "slabs_128", "kind": "slab", "nx": 128, "ny": 128, "nz": 128, "cuts": 2, "pair": "27x19",
         "forcing": "sc", "storage": "fp32", "steps": 20},
        # a run started from a snapshot on the host and saved to one
        {"name": "restart_128", "kind": "restart", "nx": 128, "ny": 128, "nz": 128, "pair": "27x19",
         "forcing": "guo", "storage": "fp32", "steps": 2},
        # records and fields of a state for analysis on the GPU
        {"name": "analysis_256", "kind": "analysis", "nx": 256, "ny": 256, "nz": 256, "pair": "27x19",
         "forcing": "sc", "storage": "fp32", "warm": 25},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _storage(rng, pair):
    return rng.choice(["fp32", "fp32", "fp16", "bf16"] if pair in ("27x19", "19x7") else ["fp32", "fp16"])


def _smooth_Re(nx, Fr):
    """A drawn lattice may be stepped a great many times: its viscosity resolves the flow (as 800 at 256^3 does) and
    stays above the growth rate of the acoustic branch."""
    return float(round(min(20 * nx / (2 * math.pi), 1000 * Fr)))


def draw(rng):
    kind = rng.choices(["cube", "box", "batch", "slab", "restart", "analysis"], [4, 3, 1, 1, 1, 1])[0]
    pair = rng.choice(["27x19", "27x19", "19x7", "19x7"] + list(PAIRS))
    forcing = rng.choice(["guo", "sc", "sc", "edm", "hcz"])
    storage = _storage(rng, pair)
    Fr = rng.choice([1.0, 0.5, 0.2])
    if kind in ("cube", "box"):
        nx = ny = nz = _log(rng, 32, 512 if kind == "cube" else 320)
        if kind == "box":
            nx, ny, nz = nx | 1 if rng.random() < 0.5 else nx, _log(rng, 17, 320), _log(rng, 17, 320)
            while nx * ny * nz > 1 << 24:
                ny, nz = max(17, ny * 3 // 4), max(17, nz * 3 // 4)
        # no more node updates than the largest listed case
        most = max(2, min(200, 20 * 512 ** 3 // (nx * ny * nz)))
        steps = _log(rng, 1, most) if rng.random() < 0.5 else rng.randint(1, most)
        Re = _smooth_Re(nx, Fr)
        return _run("", nx, ny, nz, pair, forcing, storage, steps, rng.choice(["fused", "after"]), Re, Fr)
    if kind == "batch":
        sizes = sorted({_log(rng, 32, 96) for _ in range(rng.randint(1, 4))})
        frs = rng.sample(["1", "0.7", "0.5", "0.2"], rng.randint(1, 4))
        forcings = rng.choice(["guo,sc", "guo", "sc", "edm,hcz", "guo,sc,edm,hcz"])
        return {"kind": "batch", "mode": rng.choice(["instances", "persistent", "per_step"]),
                "sizes": ",".join(map(str, sizes)), "frs": ",".join(frs), "forcings": forcings,
                "pairs": rng.choice(["19x7,27x19", "27x19", "19x7"]), "Re": 100.0, "steps": rng.randint(20, 100)}
    n = _log(rng, 32, 224)
    Re = _smooth_Re(n, Fr)
    if kind == "slab":
        return {"kind": "slab", "nx": n, "ny": _log(rng, 32, 224), "nz": _log(rng, 32, 192), "cuts": rng.randint(1, 4),
                "pair": pair, "forcing": forcing, "storage": storage, "steps": rng.randint(2, 30), "Re": Re,
                "Fr": Fr}
    if kind == "restart":
        return {"kind": "restart", "nx": n, "ny": _log(rng, 24, 160), "nz": _log(rng, 24, 160), "pair": pair,
                "forcing": forcing, "storage": storage, "steps": rng.randint(1, 4), "Re": Re, "Fr": Fr}
    return {"kind": "analysis", "nx": n, "ny": n, "nz": n, "pair": pair, "forcing": forcing, "storage": storage,
            "warm": rng.randint(2, 30), "Re": Re, "Fr": Fr}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

def _fields(nx, ny, nz, seed):
    """rho, u (3), rho' in FP64 on the GPU: the Taylor-Green velocity with one period along each side, and noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x, y, z = (torch.arange(n, dtype=torch.float64, device="cuda") * (2 * math.pi / n) for n in (nx, ny, nz))
    u = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device="cuda")
    u[0] = U0 * torch.sin(x) * torch.cos(y)[:, None] * torch.cos(z)[:, None, None]
    u[1] = -U0 * torch.cos(x) * torch.sin(y)[:, None] * torch.cos(z)[:, None, None]
    u += NOISE * U0 * (2 * torch.rand(u.shape, generator=g, dtype=torch.float64, device="cuda") - 1)
    rho = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    rho_p = 1e-2 * (2 * torch.rand(rho.shape, generator=g, dtype=torch.float64, device="cuda") - 1)
    return rho, u, rho_p


def _host(fields):
    return [f.reshape(3, -1).cpu().numpy() if f.dim() == 4 else f.reshape(-1).cpu().numpy() for f in fields]


def _params(c, nz=None):
    return lbm.lbm_params_from_physics(c["nx"], c["ny"], c["nz"] if nz is None else nz, c["pair"], c["forcing"],
                                       c.get("Re", 400.0), c.get("Fr", 0.2), 1.0, U0)


class _Lattice:
    """A simulation on a population store that the program owns."""

    def __init__(self, c, nz=None):
        self.sim = lbm.Simulation(_params(c, nz), storage=c["storage"], torch_memory=False)
        nbytes = lbm.lbm_required_bytes(self.sim.h)
        self.store = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        torch.cuda.current_stream().synchronize()
        lbm.lbm_attach(self.sim.h, self.store.data_ptr(), nbytes)
        self.pops = self.store.view(TYPES[c["storage"]])

    def __del__(self):
        self.sim.close()   # waits for the stream, then the store may go


def _is_cube(c):
    return c["nx"] == c["ny"] == c["nz"]


def _started(c, seed):
    s = _Lattice(c)
    if _is_cube(c):
        s.sim.init_tgv(seed, NOISE)
    else:
        s.sim.init_fields(*_host(_fields(c["nx"], c["ny"], c["nz"], seed)))
    return s


def _batch_specs(c):
    return [(int(n), float(fr), fo, pair) for n in c["sizes"].split(",") for fr in c["frs"].split(",")
            for fo in c["forcings"].split(",") for pair in c["pairs"].split(",")]


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"case": c}
    if kind in ("run", "analysis"):
        st["lat"] = _started(c, seed)
        if kind == "analysis":
            st["lat"].sim.step(c["warm"])
    elif kind == "restart":
        st["lat"] = _Lattice(c)
        st["fields"] = _host(_fields(c["nx"], c["ny"], c["nz"], seed))
    elif kind == "slab":
        cuts = [round(k * c["nz"] / c["cuts"]) for k in range(c["cuts"] + 1)]
        fields = _fields(c["nx"], c["ny"], c["nz"], seed)
        st["lats"] = []
        for z0, z1 in zip(cuts[:-1], cuts[1:]):
            planes = torch.arange(z0 - 1, z1 + 1, device="cuda") % c["nz"]
            s = _Lattice(c, len(planes))
            s.sim.init_fields(*_host([f[..., planes, :, :].contiguous() for f in fields]))
            st["lats"].append(s)
        st["run"] = halo.LocalSlabs([halo.LibrarySlab(s.sim) for s in st["lats"]])
    else:
        specs = _batch_specs(c)
        st["batch"] = lbm.lbm_batch_create([lbm.lbm_params_from_physics(n, n, n, pair, fo, c["Re"], fr, 1.0, U0)
                                            for n, fr, fo, pair in specs])
        st["owner"] = _Batch(st["batch"])
        lbm.lbm_batch_set_mode(st["batch"], c["mode"])
        lbm.lbm_batch_init_tgv(st["batch"], seed, NOISE)
        nodes = sum(s[0] ** 3 for s in specs)
        st["out"] = [torch.zeros(k * nodes, dtype=torch.float64, device="cuda") for k in (1, 3, 1)]
        torch.cuda.current_stream().synchronize()
    return st


class _Batch:
    def __init__(self, b):
        self.b = b

    def __del__(self):
        lbm.lbm_batch_destroy(self.b)


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------

def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "run":
        lat = state["lat"]
        if c["record"] == "fused":
            d = lat.sim.step_diagnostics(c["steps"])
        else:
            lat.sim.step(c["steps"])
            d = lat.sim.diagnostics()
        return {"record": d, "populations": lat.pops}
    if kind == "analysis":
        d = state["lat"].sim.diagnostics()
        return {"record": d, "fields": state["lat"].sim.fields_device()}
    if kind == "restart":
        sim = state["lat"].sim
        sim.init_fields(*state["fields"])
        sim.step(c["steps"])
        return {"fields": sim.fields()}
    if kind == "slab":
        state["run"].step(c["steps"])
        return {"slabs": [s.pops for s in state["lats"]]}
    b, at = state["batch"], 0
    lbm.lbm_batch_step(b, c["steps"])
    records = lbm.lbm_batch_diagnostics(b)
    for i, spec in enumerate(_batch_specs(c)):
        lbm.lbm_get_fields_device(lbm.lbm_batch_instance(b, i),
                                  *(t.data_ptr() + 8 * k * at for t, k in zip(state["out"], (1, 3, 1))))
        at += spec[0] ** 3
    return {"records": {k: torch.tensor([d[k] for d in records], dtype=torch.float32)
                        for k in ("Ek", "Ep", "eps_k", "eps_p", "eps_k_curl", "mass_f", "mass_g", "umax")},
            "fields": state["out"]}


def work(case):
    """Each population of every node read once and written once per time step; a record reads the populations
    once where no step does it; fields are 5 FP64 values per node. About 13 operations per population update."""
    c, kind = case, case["kind"]
    if kind == "batch":
        q = sum(sum(PAIRS[s[3]]) * s[0] ** 3 for s in _batch_specs(c))
        nodes = sum(s[0] ** 3 for s in _batch_specs(c))
        return {"bytes": 4 * q * (2 * c["steps"] + 2) + 40 * nodes, "flops": 13 * q * c["steps"]}
    nodes = c["nx"] * c["ny"] * c["nz"]
    pops = sum(PAIRS[c["pair"]]) * nodes
    es = BYTES[c["storage"]]
    if kind == "run":
        reads = 2 * c["steps"] + (c["record"] == "after")
        return {"bytes": pops * es * reads, "flops": 13 * pops * c["steps"]}
    if kind == "slab":
        return {"bytes": 2 * pops * es * c["steps"], "flops": 13 * pops * c["steps"]}
    if kind == "restart":
        return {"bytes": pops * es * (2 * c["steps"] + 2) + 80 * nodes, "flops": 13 * pops * (c["steps"] + 1)}
    return {"bytes": 2 * pops * es + 40 * nodes, "flops": 8 * pops}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits: full populations, two copies, plain torch
# ---------------------------------------------------------------------------------------------

def _velocities(q):
    axes = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
    edges = [(1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
    corners = [(1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)]
    es = [(0, 0, 0)]
    for e in {7: axes, 15: axes + corners, 19: axes + edges, 27: axes + edges + corners}[q]:
        es += [e, tuple(-v for v in e)]
    w = {7: (1 / 4, 1 / 8), 15: (2 / 9, 1 / 9, 0, 1 / 72), 19: (1 / 3, 1 / 18, 1 / 36),
         27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[q]
    return es, [w[sum(v * v for v in e)] for e in es], 0.25 if q == 7 else 1.0 / 3.0


def _dot(e, u):
    parts = [u[a] if v > 0 else -u[a] for a, v in enumerate(e) if v]
    return sum(parts[1:], parts[0]) if parts else 0.0


class _Equilibrium:
    """w rho (1 + e.u / c^2 + (e.u)^2 / (2 c^4) - u^2 / (2 c^2)) of every velocity."""

    def __init__(self, rho, u, velocity_set):
        self.es, self.ws, self.cs2 = velocity_set
        self.rho, self.u = rho, u
        self.rest = rho * (1.0 - (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) / (2 * self.cs2))

    def __call__(self, i):
        eu = _dot(self.es[i], self.u) / self.cs2
        return self.ws[i] * (self.rest + self.rho * eu * (1.0 + 0.5 * eu)) if i else self.ws[0] * self.rest


def _moved(t, e):
    return torch.roll(t, (e[2], e[1], e[0]), (-3, -2, -1)) if any(e) else t


class _Exact:
    """Section 2 of the paper with the library's default readings, in FP64, for some Froude numbers at once."""

    def __init__(self, nx, pair, forcing, Re, frs):
        qf, qg = PAIRS[pair]
        self.forcing, self.f_set, self.g_set = forcing, _velocities(qf), _velocities(qg)
        L = nx / (2 * math.pi)
        self.nu = self.D = U0 * L / Re
        self.tau_f, self.tau_g = self.nu / self.f_set[2] + 0.5, self.D / self.g_set[2] + 0.5
        self.N = torch.tensor([U0 / (fr * L) for fr in frs], dtype=torch.float64, device="cuda").reshape(-1, 1, 1, 1)
        self.G, self.beta = self.N / 1024.0, -self.N * 1024.0
        self.steps = 0

    def start(self, rho, u, rho_p):
        n = len(self.N)
        f = _Equilibrium(rho, u, self.f_set)
        g = _Equilibrium(rho_p + 1.0, u, self.g_set)
        self.f = [f(i).expand(n, *rho.shape) for i in range(len(self.f_set[0]))]
        self.g = [g(i).expand(n, *rho.shape) for i in range(len(self.g_set[0]))]

    def macro(self):
        es = self.f_set[0]
        rho = sum(self.f[1:], self.f[0])
        j = [sum(e[a] * self.f[i] for i, e in enumerate(es) if e[a]) for a in range(3)]
        a = sum(self.g[1:], self.g[0]) - 1.0
        kappa = -0.5 * (1 - 1 / (2 * self.tau_g)) * self.beta
        rho_p = (a + kappa * j[2] / rho) / (1 + kappa * self.G / (2 * rho))
        fz = -self.G * rho_p
        return rho, j, rho_p, fz, [j[0] / rho, j[1] / rho, (j[2] + 0.5 * fz) / rho]

    def step(self):
        rho, j, rho_p, fz, u = self.macro()
        es, ws, cs2 = self.f_set
        tau, pref = self.tau_f, 1 - 1 / (2 * self.tau_f)
        v = u
        if self.forcing in ("sc", "edm"):
            v = [j[0] / rho, j[1] / rho, (j[2] + (tau * fz if self.forcing == "sc" else 0.0)) / rho]
        eq = _Equilibrium(rho, v, self.f_set)
        eq2 = _Equilibrium(rho, [v[0], v[1], v[2] + fz / rho], self.f_set) if self.forcing == "edm" else None
        for i, e in enumerate(es):
            feq = eq(i)
            new = self.f[i] - (self.f[i] - feq) / tau
            if self.forcing == "guo":
                new += pref * ws[i] * ((e[2] - u[2]) / cs2 + _dot(e, u) * e[2] / cs2 ** 2) * fz
            elif self.forcing == "hcz":
                new += pref * (e[2] - u[2]) * fz / (rho * cs2) * feq
            elif self.forcing == "edm":
                new += eq2(i) - feq
            self.f[i] = _moved(new, e)
        es, ws, _ = self.g_set
        eq = _Equilibrium(rho_p + 1.0, u, self.g_set)
        source = -u[2] * self.beta
        for i, e in enumerate(es):
            self.g[i] = _moved(self.g[i] - (self.g[i] - eq(i)) / self.tau_g + ws[i] * source, e)
        self.steps += 1

    def records(self):
        """The averages that need no closure, one value per Froude number."""
        rho, _, rho_p, _, u = self.macro()
        n3, gn2 = rho[0].numel(), 2.0 ** -20

        def total(t):
            return t.sum((-3, -2, -1))

        def d(t, axis):   # along x, y, z
            return 0.5 * (torch.roll(t, -1, -1 - axis) - torch.roll(t, 1, -1 - axis))
        usq = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        curl = (d(u[2], 1) - d(u[1], 2)) ** 2 + (d(u[0], 2) - d(u[2], 0)) ** 2 + (d(u[1], 0) - d(u[0], 1)) ** 2
        return {"Ek": 0.5 * total(usq) / n3, "Ep": 0.5 * gn2 * total(rho_p ** 2) / n3,
                "eps_p": self.D * gn2 * total(d(rho_p, 0) ** 2 + d(rho_p, 1) ** 2 + d(rho_p, 2) ** 2) / n3,
                "eps_k_curl": self.nu * total(curl) / n3, "mass_f": total(rho), "mass_g": total(sum(self.g[1:], self.g[0])),
                "umax": usq.amax((-3, -2, -1)).sqrt()}

    def record(self):
        return {**{k: None for k in _KEYS}, **{k: float(v[0]) for k, v in self.records().items()}, "step": self.steps}

    def store(self, storage):
        """The natural store layout: deviations slot by slot, 16-bit rows of even length in half-row order."""
        out = torch.stack([f[0] - w for f, w in zip(self.f, self.f_set[1])] +
                          [g[0] - w for g, w in zip(self.g, self.g_set[1])])
        nx = out.shape[-1]
        if BYTES[storage] == 2 and nx % 2 == 0:
            out = torch.stack([out[..., :nx // 2], out[..., nx // 2:]], -1)
        return out.reshape(-1)


_KEYS = ("Ek", "Ep", "eps_k", "eps_p", "eps_k_curl", "mass_f", "mass_g", "mom_x", "mom_y", "mom_z", "umax", "step",
         "t", "Ek_phys", "Ep_phys", "eps_k_phys", "eps_p_phys", "eps_k_curl_phys")


def _tgv(n, seed):
    """Equation 20 with the library's documented noise: SplitMix64 draws in [-1, 1) by component and node."""
    dev = "cuda"
    x = torch.arange(n, dtype=torch.float64, device=dev) * (2 * math.pi / n)
    u = torch.zeros((3, n, n, n), dtype=torch.float64, device=dev)
    u[0] = U0 * torch.sin(x) * torch.cos(x)[:, None] * torch.cos(x)[:, None, None]
    u[1] = -U0 * torch.cos(x) * torch.sin(x)[:, None] * torch.cos(x)[:, None, None]

    def i64(v):
        return v - (1 << 64) if v >= 1 << 63 else v

    def shr(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)
    for a in range(3):
        z = torch.arange(a * n ** 3 + 1, (a + 1) * n ** 3 + 1, dtype=torch.int64, device=dev)
        z = z * i64(0x9E3779B97F4A7C15) + seed
        z = (z ^ shr(z, 30)) * i64(0xBF58476D1CE4E5B9)
        z = (z ^ shr(z, 27)) * i64(0x94D049BB133111EB)
        z = z ^ shr(z, 31)
        u[a] += NOISE * U0 * (shr(z, 11).double() * (2.0 ** -52) - 1.0).reshape(n, n, n)
    one = torch.ones((n, n, n), dtype=torch.float64, device=dev)
    return one, u, torch.zeros_like(one)


def _known(record, c):
    """In 16 bits the density perturbation, which grows from zero, is the storage's own rounding at first."""
    return {**record, "Ep": None, "eps_p": None} if BYTES[c["storage"]] == 2 else record


def _advanced(c, start, frs, steps):
    e = _Exact(c["nx"], c["pair"], c["forcing"], c.get("Re", 400.0), frs)
    e.start(*start)
    first = e.record() if steps and len(frs) == 1 else None
    for _ in range(steps):
        e.step()
    return e, first


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        return _exact_batch(c, seed)
    nodes, steps = c["nx"] * c["ny"] * c["nz"], c.get("steps", c.get("warm", 0))
    if kind == "slab" or nodes > 300 ** 3 or nodes * steps > 1.9e9:
        # a slab's store also holds the ghost planes, whatever the exchange left there
        return None
    cube = _is_cube(c) and kind != "restart"
    start = _tgv(c["nx"], seed) if cube else _fields(c["nx"], c["ny"], c["nz"], seed)
    e, first = _advanced(c, start, [c.get("Fr", 0.2)], steps)
    if kind == "run":
        # an odd step count leaves the store in the other layout of the in-place streaming
        return {"record": _known(first if c["record"] == "fused" else e.record(), c),
                "populations": e.store(c["storage"]) if steps % 2 == 0 else None}
    rho, _, rho_p, _, u = e.macro()
    fields = [rho.reshape(-1), torch.stack(u).reshape(3, -1), rho_p.reshape(-1)]
    if kind == "analysis":
        return {"record": _known(e.record(), c), "fields": fields[:2] + [fields[2] if c["storage"] == "fp32" else None]}
    return {"fields": [t.cpu().numpy() for t in fields]}


def _exact_batch(c, seed):
    specs = _batch_specs(c)
    groups = sorted({(n, fo, pair) for n, _, fo, pair in specs})
    if len(groups) * c["steps"] > 2400 or sum(s[0] ** 3 for s in specs) * c["steps"] > 3e9:
        return None
    at, where = 0, {}
    for s in specs:
        where[s] = at
        at += s[0] ** 3
    out = [torch.zeros(k * at, dtype=torch.float64, device="cuda") for k in (1, 3, 1)]
    records = {k: torch.zeros(len(specs), dtype=torch.float64) for k in
               ("Ek", "Ep", "eps_p", "eps_k_curl", "mass_f", "mass_g", "umax")}
    for n, fo, pair in groups:
        frs = [s[1] for s in specs if (s[0], s[2], s[3]) == (n, fo, pair)]
        e, _ = _advanced({"nx": n, "pair": pair, "forcing": fo, "Re": c["Re"]}, _tgv(n, seed), frs, c["steps"])
        rho, _, rho_p, _, u = e.macro()
        recs = e.records()
        for b, fr in enumerate(frs):
            s = (n, fr, fo, pair)
            for t, k, v in zip(out, (1, 3, 1), (rho[b], torch.stack([w[b] for w in u]), rho_p[b])):
                t[k * where[s]:k * (where[s] + n ** 3)] = v.reshape(-1)
            for k, v in recs.items():
                records[k][specs.index(s)] = float(v[b])
    return {"records": {**records, "eps_k": None}, "fields": out}
