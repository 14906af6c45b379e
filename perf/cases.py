"""The work a user has this library do, as measurable cases.

Every case goes through the package's public entry points: a
:class:`~paper_1703_00185_gb300.Lattice` set up, advanced and read out, a
:class:`~paper_1703_00185_gb300.Batch` of lattices, the allocation-free batch
call, the job server, and a restart from host populations.  Sizes are those of
the benchmark (2048 x 8192), of the paper's table (1024 x 8192), of the parity
case (256 x 128), of the batched and serving workloads, and odd ones as the
tests use.  ``exact`` is the same method in plain torch, 64 bits, written from
its definition.
"""
import math

import numpy as np
import torch

import paper_1703_00185_gb300 as lbm
from paper_1703_00185_gb300 import serving

# ---------------------------------------------------------------- the cases

LISTED = [
    # the benchmark lattice: a production run advances it in bursts and reads the fields
    {"name": "run_fp64_2048x8192", "kind": "run", "Lx": 2048, "Ly": 8192, "precision": "fp64", "steps": 8,
     "tau": 0.8},
    # the same in FP32 storage with double-float wide terms, the form for throughput
    {"name": "run_fp32df_2048x8192", "kind": "run", "Lx": 2048, "Ly": 8192, "precision": "fp32-df", "steps": 8,
     "tau": 0.8},
    # FP32 storage with FP64 wide terms on the lattice of the paper's table
    {"name": "run_fp32_1024x8192", "kind": "run", "Lx": 1024, "Ly": 8192, "precision": "fp32", "steps": 8,
     "tau": 0.8},
    # the parity case, which stays in L2: a small study, replayed graphs on a stream of its own
    {"name": "run_fp64_256x128_graph", "kind": "run", "Lx": 256, "Ly": 128, "precision": "fp64", "steps": 100,
     "tau": 0.8, "own_stream": True},
    # one step and a look at the fields, on an odd size: a monitoring loop, all latency and launches
    {"name": "monitor_fp64_130x257", "kind": "run", "Lx": 130, "Ly": 257, "precision": "fp64", "steps": 1,
     "tau": 0.8},
    # the schedule of separate kernels (propagate, bc, collide), a ragged lattice
    {"name": "separate_fp64_1000x2050", "kind": "run", "Lx": 1000, "Ly": 2050, "precision": "fp64", "steps": 4,
     "tau": 0.8, "kernel": "separate"},
    # a new initial state on a lattice that is there already, and its first step: every run and every
    # served job begins so
    {"name": "init_fp64_1024x4096", "kind": "init", "Lx": 1024, "Ly": 4096, "precision": "fp64", "steps": 1,
     "tau": 0.8},
    # 64 uneven lattices that share tau and g (the batched workload), launch shape from the autotuner
    {"name": "batch_fp64_64", "kind": "batch", "n": 64, "precision": "fp64", "steps": 16, "lo": 128, "hi": 1024,
     "sizes": 1, "sweep": False, "tune": True},
    # a sweep over tau and g on 100 middling lattices, odd sizes, default launch shape
    {"name": "sweep_fp64_100", "kind": "batch", "n": 100, "precision": "fp64", "steps": 16, "lo": 60, "hi": 400,
     "sizes": 2, "sweep": True, "tune": False},
    # the batch call that allocates nothing, FP32 storage, as a loop of a host program makes it
    {"name": "static_fp32df_24", "kind": "static", "n": 24, "precision": "fp32-df", "steps": 16, "lo": 64, "hi": 512,
     "sizes": 3, "sweep": True},
    # a burst of jobs of both precisions through the server, results fetched to the host
    {"name": "serve_12_jobs", "kind": "serve", "n": 12, "lo": 32, "hi": 400, "sizes": 4, "steps": 150},
    # a restart: populations up from pinned host memory, some steps, populations back down
    {"name": "restart_fp32df_512x1024", "kind": "restart", "Lx": 512, "Ly": 1024, "precision": "fp32-df",
     "steps": 4, "tau": 0.7},
]


def listed():
    return [dict(c) for c in LISTED]


def _log(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same kinds with sizes over their whole ranges; at most as
    many site updates as the 64 uneven lattices take."""
    kind = rng.choice(["run", "run", "run", "run", "init", "batch", "static", "serve", "restart"])
    tau = round(rng.uniform(0.6, 1.4), 3)
    precision = rng.choice(["fp64", "fp64", "fp32-df", "fp32"])
    if kind == "run":
        Lx, Ly = _log(rng, 16, 2048), _log(rng, 16, 8192)
        c = {"kind": kind, "Lx": Lx, "Ly": Ly, "precision": precision,
             "steps": 1 if rng.random() < 0.2 else _log(rng, 2, 100 if Lx * Ly < 1 << 20 else 8), "tau": tau}
        if rng.random() < 0.3:
            c["own_stream"] = True
        if rng.random() < 0.2:
            c["kernel"] = "separate"
        return c
    if kind == "init":
        return {"kind": kind, "Lx": _log(rng, 16, 2048), "Ly": _log(rng, 16, 4096), "precision": precision, "steps": 1,
                "tau": tau}
    if kind == "serve":
        return {"kind": kind, "n": rng.randint(3, 16), "lo": 16, "hi": _log(rng, 64, 500),
                "sizes": rng.randrange(1 << 20), "steps": _log(rng, 10, 150)}
    if kind == "restart":
        return {"kind": kind, "Lx": _log(rng, 16, 700), "Ly": _log(rng, 16, 1100), "precision": precision,
                "steps": rng.randint(1, 6), "tau": tau}
    hi = _log(rng, 64, 640)
    c = {"kind": kind, "n": rng.randint(2, 100), "precision": precision, "steps": rng.randint(2, 16), "lo": 12,
         "hi": hi, "sizes": rng.randrange(1 << 20), "sweep": rng.random() < 0.5}
    if kind == "batch":
        c["tune"] = rng.random() < 0.3
    return c


def _lattices(case):
    """Size and parameters of each lattice of a batch or of each job, from the
    case alone (per-lattice seeds come from the seed of the inputs)."""
    rng = np.random.default_rng(case["sizes"])
    n, lo, hi = case["n"], case["lo"], case["hi"]
    if case["sizes"] == 1:  # the batched workload's size classes
        Lx, Ly = rng.choice(np.arange(lo, hi + 1, 128), n), rng.choice(np.arange(2 * lo, 2 * hi + 1, 256), n)
    else:
        Lx = np.exp(rng.uniform(math.log(lo), math.log(hi + 1), n)).astype(int)
        Ly = np.exp(rng.uniform(math.log(lo), math.log(2 * hi + 1), n)).astype(int)
    T_bot = rng.uniform(1.2, 1.8, n)
    tau, g0 = rng.uniform(0.6, 1.2, n), rng.uniform(0.0, 2e-4, n)
    steps = rng.integers(max(1, case["steps"] // 3), case["steps"] + 1, n)
    fp64 = rng.random(n) < 0.5
    out = []
    for i in range(n):
        sweep = case.get("sweep", False)
        out.append({"Lx": max(3, int(Lx[i])), "Ly": max(6, int(Ly[i])), "T_bot": float(T_bot[i]),
                    "tau": float(tau[i]) if sweep else 0.8, "g0": float(g0[i]) if sweep else 1e-4,
                    "steps": int(steps[i]) if case["kind"] == "serve" else case["steps"],
                    "precision": case.get("precision") or ("fp64" if fp64[i] else "fp32-df")})
    return out


# ------------------------------------------------------- preparing and running

class _Single:
    """A lattice with a state."""

    def __init__(self, case, seed):
        self.case, self.seed = case, seed
        stream = torch.cuda.Stream() if case.get("own_stream") else None
        self.lat = lbm.Lattice(case["Lx"], case["Ly"], tau=case["tau"], precision=case["precision"],
                               kernel=case.get("kernel", "fused"), stream=stream)
        if case["kind"] == "restart":
            f = _restart_populations(case, seed).to("cpu")
            self.up = f.pin_memory()
            self.down = torch.empty_like(self.up).pin_memory()
        else:
            self.lat.init_rayleigh_taylor(seed)

    def run(self):
        lat, case = self.lat, self.case
        if case["kind"] == "restart":
            lat.set_populations(self.up)
            lat.step(case["steps"])
            return lat.populations(out=self.down)
        if case["kind"] == "init":
            lat.init_rayleigh_taylor(self.seed)
        if not case.get("own_stream"):
            lat.step(case["steps"])
            return lat.fields_device()
        here = torch.cuda.current_stream()
        lat.stream.wait_stream(here)
        with torch.cuda.stream(lat.stream):
            lat.step(case["steps"])
            out = lat.fields_device()
        here.wait_stream(lat.stream)
        for t in out:
            t.record_stream(here)
        return out


def _gather(fields):
    """The fields of many lattices, one array per field, the lattices one after another."""
    return [torch.cat([v.reshape(-1) for v in parts]) for parts in zip(*fields)]


class _Many:
    """A batch of lattices with states."""

    def __init__(self, case, seed):
        self.case = case
        self.lats = []
        for i, j in enumerate(_lattices(case)):
            lat = lbm.Lattice(j["Lx"], j["Ly"], tau=j["tau"], g0=j["g0"], T_bot=j["T_bot"],
                              precision=j["precision"])
            lat.init_rayleigh_taylor(1000 * seed + i)
            self.lats.append(lat)
        self.batch = lbm.Batch(self.lats)
        if case["tune"]:
            self.batch.autotune(trial_steps=3, use_cache=False)

    def run(self):
        self.batch.step(self.case["steps"])
        self.batch.synchronize()
        return _gather([lat.fields_device() for lat in self.lats])


class _Static:
    """Lattices in device memory of the caller's own, stepped by the call that allocates nothing."""

    def __init__(self, case, seed):
        self.case, self.h = case, []
        self.jobs = _lattices(case)
        self.stream = torch.cuda.current_stream().cuda_stream
        self.mem = []
        for i, j in enumerate(self.jobs):
            p = lbm.lbm_default_params()
            p.tau, p.g0, p.T_bot, p.precision = j["tau"], j["g0"], j["T_bot"], lbm.PRECISIONS[j["precision"]]
            nbytes = lbm.lbm_required_bytes(j["Lx"], j["Ly"], p)
            mem = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
            h = lbm.lbm_create_ext(j["Lx"], j["Ly"], p, mem.data_ptr(), nbytes, self.stream)
            lbm.lbm_init_rayleigh_taylor(h, 1000 * seed + i)
            self.mem.append(mem)
            self.h.append(h)

    def run(self):
        lbm.lbm_batch_step_static(self.h, self.case["steps"], self.stream)
        out = []
        for j, h in zip(self.jobs, self.h):
            rho = torch.empty((j["Lx"], j["Ly"]), dtype=torch.float64, device="cuda")
            u = torch.empty((2, j["Lx"], j["Ly"]), dtype=torch.float64, device="cuda")
            T = torch.empty_like(rho)
            lbm.lbm_fields_device(h, rho, u, T)
            out.append((rho, u, T))
        return _gather(out)

    def __del__(self):
        for h in self.h:
            lbm.lbm_destroy(h)


class _Serve:
    """A running server and a burst of jobs to come."""

    def __init__(self, case, seed):
        self.jobs = [dict(j, seed=1000 * seed + i) for i, j in enumerate(_lattices(case))]
        self.server = serving.Server(4 << 30, max_steps_per_tick=16)

    def run(self):
        srv = self.server
        ids = [srv.submit(j["Lx"], j["Ly"], j["steps"], j["precision"], j["seed"], T_bot=j["T_bot"])
               for j in self.jobs]
        left, got = set(ids), {}
        while left:
            srv.tick()
            for jid in srv.poll():
                got[jid] = srv.fetch(jid)
                left.discard(jid)
        return [np.concatenate([a.reshape(-1) for a in parts]) for parts in zip(*(got[jid] for jid in ids))]

    def __del__(self):
        if hasattr(self, "server"):
            self.server.close()


def prepare(case, seed):
    kind = {"run": _Single, "init": _Single, "restart": _Single, "batch": _Many, "static": _Static,
            "serve": _Serve}[case["kind"]]
    return kind(case, seed)


def run(state):
    return state.run()


# ------------------------------------------------------------- work, tolerance

def work(case):
    """Bytes: per step every population of every site read and written once
    (37 values each way, 8 bytes or 4 in FP32 storage), and for a read-out the
    37 values read and the 4 FP64 fields written.  FLOPs: 2354 per site update,
    the collision written plainly."""
    bytes_, flops = 0.0, 0.0

    def add(sites, steps, precision, fields=True):
        nonlocal bytes_, flops
        e = 8 if precision == "fp64" else 4
        bytes_ += sites * (74.0 * e * steps + (37.0 * e + 32.0 if fields else 0.0))
        flops += sites * (2354.0 * steps + (200.0 if fields else 0.0))

    if case["kind"] in ("batch", "static", "serve"):
        for j in _lattices(case):
            add(j["Lx"] * j["Ly"], j["steps"], j["precision"])
            if case["kind"] == "serve":  # the initial state
                bytes_ += j["Lx"] * j["Ly"] * 37.0 * (8 if j["precision"] == "fp64" else 4)
    else:
        sites = case["Lx"] * case["Ly"]
        add(sites, case.get("steps", 0), case["precision"], fields=case["kind"] != "restart")
        if case["kind"] == "restart":  # FP64 populations up and down
            bytes_ += 2 * sites * 37.0 * 8
        if case["kind"] == "init":
            bytes_ += sites * 37.0 * (8 if case["precision"] == "fp64" else 4)
            flops += sites * 150.0
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """About four times the distance to ``exact`` that the parent of this file
    showed.  The velocity decides: it grows from nothing, so that its error is a
    rounding of the O(1) populations over a small number (one step 5e-14, up to
    16 steps 3e-13, 150 steps 1.2e-12 in FP64; 1.3e-5 in FP32 storage).
    Populations themselves: 1e-15 and 3.4e-8."""
    fp64 = case.get("precision") == "fp64"
    if case["kind"] == "restart":
        return {"rel": 5e-15 if fp64 else 1.5e-7, "max": 5e-13 if fp64 else 1e-5}
    if not fp64:  # the burst of jobs holds both precisions
        return {"rel": 5e-5, "max": 5e-4}
    if case["steps"] == 1:
        return {"rel": 2e-13, "max": 2e-12}
    return {"rel": 1.2e-12 if case["steps"] <= 16 else 5e-12, "max": 1e-11 if case["steps"] <= 16 else 4e-11}


# ----------------------------------------------------- the method in 64 bits

# The D2Q37 quadrature: thermal speed s and the weights of the shells
# |c|^2 = 0, 1, 2, 4, 5, 8, 9, 10 that make every Gaussian moment up to degree 9 exact.
S = 1.1969797703930745
W_SHELL = {0: 0.2331506691323525, 1: 0.107306091542219, 2: 0.05766785988879488, 4: 0.01420821615845075,
           5: 0.005353049000513775, 8: 0.0010119375926735754, 9: 0.00024530102775771736, 10: 0.00028341425299419824}
T_TOP, T_BOT, G0 = 0.5, 1.5, 1e-4  # the entry points' defaults
CHUNK = 1 << 19  # sites of one piece of a collision (the temporaries hold 37 values a site)


def _velocities():
    """Hops in the library's population order, which a host array of populations follows."""
    cx, cy = lbm.lbm_velocity_set()
    return [int(v) for v in cx], [int(v) for v in cy]


class _Method:
    def __init__(self, device):
        self.cx, self.cy = _velocities()
        t = dict(dtype=torch.float64, device=device)
        self.X = S * torch.tensor(self.cx, **t)[:, None]
        self.Y = S * torch.tensor(self.cy, **t)[:, None]
        self.W = torch.tensor([W_SHELL[a * a + b * b] for a, b in zip(self.cx, self.cy)], **t)[:, None]
        self.X2 = self.X * self.X + self.Y * self.Y

    def equilibrium(self, rho, ux, uy, T):
        """The Maxwellian's Hermite expansion to 4th order, [37, n]."""
        a = self.X * ux + self.Y * uy
        q, th, x2 = ux * ux + uy * uy, T - 1.0, self.X2
        P = (1.0 + a + 0.5 * (a * a - q + th * (x2 - 2.0)) + a * (a * a - 3.0 * q + 3.0 * th * (x2 - 4.0)) / 6.0
             + (a ** 4 - 6.0 * a * a * q + 3.0 * q * q + 6.0 * th * (a * a * (x2 - 6.0) + q * (4.0 - x2))
                + 3.0 * th * th * (x2 * x2 - 8.0 * x2 + 8.0)) / 24.0)
        return self.W * rho * P

    def moments(self, f):
        rho = f.sum(0)
        ux, uy = (self.X * f).sum(0) / rho, (self.Y * f).sum(0) / rho
        return rho, ux, uy, (((self.X - ux) ** 2 + (self.Y - uy) ** 2) * f).sum(0) / (2.0 * rho)

    def fields(self, f):
        parts = [self.moments(p) for p in f.reshape(37, -1).split(CHUNK, dim=1)]
        rho, ux, uy, T = (torch.cat(v).reshape(f.shape[1:]) for v in zip(*parts))
        return rho, torch.stack([ux, uy]), T

    def step(self, f, tau, g0, T_top, T_bot):
        """Pull with periodic x, diffuse walls that give back each column's leaving mass, BGK collision."""
        Ly = f.shape[2]
        g = torch.zeros_like(f)
        for l, (cx, cy) in enumerate(zip(self.cx, self.cy)):
            moved = torch.roll(f[l], cx, dims=0)
            if cy >= 0:
                g[l, :, cy:] = moved[:, :Ly - cy]
            else:
                g[l, :, :cy] = moved[:, -cy:]
        one = torch.ones(1, dtype=f.dtype, device=f.device)
        for rows, Tw in ((range(3), T_bot), (range(Ly - 3, Ly), T_top)):
            fw = self.equilibrium(one, 0 * one, 0 * one, Tw * one)[:, 0]
            gone = [(l, y) for y in rows for l in range(37) if not 0 <= y - self.cy[l] < Ly]
            out = sum(f[l, :, y] for y in rows for l in range(37) if not 0 <= y + self.cy[l] < Ly)
            rho_w = out / sum(fw[l] for l, _ in gone)
            for l, y in gone:
                g[l, :, y] = rho_w * fw[l]
        flat = g.reshape(37, -1)
        for p in flat.split(CHUNK, dim=1):
            rho, ux, uy, T = self.moments(p)
            p -= (p - self.equilibrium(rho, ux, uy - tau * g0, T - 0.5 * (tau * g0) ** 2)) / tau
        return g

    def rayleigh_taylor(self, Lx, Ly, seed, T_top, T_bot):
        """Cold over hot, a sine of amplitude Ly / 64 between them, 0.1 % noise from SplitMix64."""
        with np.errstate(over="ignore"):
            z = np.uint64(seed) + np.arange(Lx * Ly, dtype=np.uint64) + np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
        U = (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
        yi = 0.5 * Ly + (Ly / 64.0) * np.sin(2.0 * np.pi * (np.arange(Lx) + 0.5) / Lx)
        T0 = np.where((np.arange(Ly) + 0.5)[None, :] < yi[:, None], T_bot, T_top)
        T = torch.from_numpy((T0.reshape(-1) * (1.0 + 1e-3 * (2.0 * U - 1.0)))).to(self.X.device)
        f = torch.empty((37, Lx * Ly), dtype=torch.float64, device=T.device)
        for p, t in zip(f.split(CHUNK, dim=1), T.split(CHUNK)):
            p.copy_(self.equilibrium(1.0 / t, 0 * t, 0 * t, t))
        return f.reshape(37, Lx, Ly)


def _restart_populations(case, seed):
    """Populations of a developed flow: equilibria of smooth fields with noise
    off equilibrium, in the library's order, [37, Lx, Ly] float64 on the GPU."""
    m = _Method("cuda")
    Lx, Ly = case["Lx"], case["Ly"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.arange(Lx, dtype=torch.float64, device="cuda")[:, None] / Lx * 2 * math.pi
    y = torch.arange(Ly, dtype=torch.float64, device="cuda")[None, :] / Ly
    ph = torch.rand(4, generator=gen, dtype=torch.float64, device="cuda") * 2 * math.pi
    T = T_BOT + (T_TOP - T_BOT) * y + 0.05 * torch.sin(x + ph[0])
    ux = 0.04 * torch.sin(2 * x + ph[1]) * torch.sin(math.pi * y)
    uy = 0.04 * torch.sin(x + ph[2]) * torch.sin(math.pi * y)
    rho = 1.0 / T * (1.0 + 0.02 * torch.sin(3 * x + ph[3]))
    n = Lx * Ly
    f = torch.empty((37, n), dtype=torch.float64, device="cuda")
    fields = [v.expand(Lx, Ly).reshape(-1) for v in (rho, ux, uy, T)]
    for p, r, a, b, t in zip(f.split(CHUNK, dim=1), *(v.split(CHUNK) for v in fields)):
        p.copy_(m.equilibrium(r, a, b, t))
    noise = torch.rand((37, n), generator=gen, dtype=torch.float64, device="cuda")
    return (f * (1.0 + 1e-3 * (2.0 * noise - 1.0))).reshape(37, Lx, Ly)


def exact(case, seed):
    m = _Method("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] in ("batch", "static", "serve"):
        jobs = _lattices(case)
        if sum(j["steps"] for j in jobs) > 1700:  # some 5 ms a step of a small lattice
            return None
        out = []
        for i, j in enumerate(jobs):
            f = m.rayleigh_taylor(j["Lx"], j["Ly"], 1000 * seed + i, T_TOP, j["T_bot"])
            for _ in range(j["steps"]):
                f = m.step(f, j["tau"], j["g0"], T_TOP, j["T_bot"])
            out.append(m.fields(f))
        out = _gather(out)
        return [v.cpu().numpy() for v in out] if case["kind"] == "serve" else out
    if case["kind"] == "restart":
        f = _restart_populations(case, seed).to(m.X.device)
    else:
        f = m.rayleigh_taylor(case["Lx"], case["Ly"], seed, T_TOP, T_BOT)
    for _ in range(case.get("steps", 0)):
        f = m.step(f, case["tau"], G0, T_TOP, T_BOT)
    if case["kind"] == "restart":
        return f.cpu()
    return m.fields(f)
