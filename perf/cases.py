"""What is timed of this package: stepping beds of the sizes, storages and models that its
workloads, tests and benchmark use, reading the results back, serving many beds at once, and
the cell binning on device arrays.

A pass steps a bed through the Python binding of the C ABI and reads back what such a user wants
of it (particles, gas fields, per-step statistics, spins).  The gas arithmetic of a bed stored in
32 or 16 bits is in FP32 although the library exports it as FP64, so those outputs are kept in
FP32, as a program that stores them would; positions are accumulated in FP64 and stay FP64.
Beds of up to RESTART_CELLS cells start every pass from the same state (loading it costs little
there); larger ones go on from where the pass before left them, as a long run does.

``exact`` restates the coupled step in FP64 with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_1303_2653_gb300 import lbdps as L
from paper_1303_2653_gb300 import workloads as W

STORAGE = {"f64": W.STORE_F64, "f32": W.STORE_F32, "f16": W.STORE_F16, "bf16": W.STORE_BF16}
POP_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
RESTART_CELLS = 1 << 16


# ------------------------------------------------------------------ the cases

def _bed(bed, n, particles, storage, steps, les=0.0, read="particles", **more):
    case = {"what": "bed", "bed": bed, "nx": n[0], "ny": n[1], "particles": particles,
            "storage": storage, "steps": steps, "les": les, "read": read}
    if len(n) == 3:
        case["nz"] = n[2]
    case.update(more)
    return case


def listed():
    return [
        # the smallest calls: one jet bed in FP64 (2,000 particles, walls, inlet and outlet),
        # bound by launches and dependent loads; every field a plot of the bed needs
        dict(_bed("bubbling", (64, 128), 2000, "f64", 100, read="particles fields"),
             name="bubbling 64x128 f64"),
        # the binning that graph-capturing hosts call on their own buffers, at the 2D riser's size
        {"name": "binning 256x2048", "what": "binning", "nx": 256, "ny": 2048, "particles": 200000},
        # a small section with odd sides (partly filled warps and tiles), every step's statistics
        # taken, Smagorinsky model on as in every served bed
        dict(_bed("riser2d", (75, 193), 5521, "f32", 50, les=0.1, read="particles monitored"),
             name="riser 75x193 f32 les"),
        # the 2D riser of the benchmark: the ordinary call
        dict(_bed("riser2d", (256, 2048), 200000, "f32", 64, read="particles fields"),
             name="riser 256x2048 f32"),
        # the largest served lattice in 16-bit storage
        dict(_bed("riser2d", (512, 2048), 400000, "f16", 64, les=0.1, read="particles fields"),
             name="riser 512x2048 f16 les"),
        # the circulating riser of Table 2: three particles per cell, inlet and outlet, rows of 60
        dict(_bed("cfb", (60, 720), 123921, "f32", 64, les=0.1, read="particles fields"),
             name="circulating 60x720 f32 les"),
        # the dense soft-sphere bed (about 11 particles per cell, most of them in contact)
        dict(_bed("packed", (256, 1024), 1460252, "f32", 16, les=0.1), name="packed 256x1024 f32"),
        # soft spheres with friction in 3D: spins carried, about 80 particles per cell
        dict(_bed("packed", (16, 16, 32), 342247, "f32", 16, friction=True, read="particles spin"),
             name="packed 16x16x32 friction"),
        # a 3D section with odd sides in the other 16-bit storage, Smagorinsky model on
        dict(_bed("riser3d", (100, 75, 333), 148860, "bf16", 32, les=0.1),
             name="riser 100x75x333 bf16 les"),
        # a snapshot of a 3D bed: a few steps, then all gas fields and the particles
        dict(_bed("riser3d", (96, 96, 192), 105469, "f32", 8, read="particles fields all"),
             name="snapshot 96x96x192 f32"),
        # the largest: the 3D riser of the benchmark with every step's statistics
        dict(_bed("riser3d", (256, 256, 1024), 4000000, "f32", 20, read="particles monitored"),
             name="riser 256x256x1024 f32"),
        # independent beds of the serving stream's kinds and sizes, submitted together, each
        # one's particles taken at its end
        {"name": "serving 24", "what": "serving", "requests": 24, "steps": 200},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    what = rng.choice(["riser2d", "riser2d", "riser2d", "riser3d", "riser3d", "bubbling", "cfb",
                       "packed", "packed3", "binning", "serving"])
    les = rng.choice([0.0, 0.1])
    if what == "binning":
        nx, ny = int(_log(rng, 32, 512)), int(_log(rng, 64, 2048))
        return {"what": "binning", "nx": nx, "ny": ny,
                "particles": int(_log(rng, 1000, max(2000, nx * ny * 0.9)))}
    if what == "serving":
        return {"what": "serving", "requests": rng.randint(8, 24), "steps": rng.randint(64, 200)}
    if what == "bubbling":
        nx = int(_log(rng, 32, 256))
        ny = int(_log(rng, 64, min(512, RESTART_CELLS // nx)))
        return _bed("bubbling", (nx, ny), int(nx * ny * rng.uniform(0.1, 0.5)),
                    rng.choice(["f64", "f32", "f16"]), rng.randint(40, 100), 0.1,
                    "particles fields")
    if what == "cfb":
        nx = int(_log(rng, 20, 120))
        ny = int(_log(rng, 100, min(1000, RESTART_CELLS // nx)))
        return _bed("cfb", (nx, ny), int(nx * ny * rng.uniform(1.0, 2.87)), "f32",
                    rng.randint(20, 64), 0.1, "particles fields")
    if what == "packed":
        nx, ny = int(_log(rng, 48, 256)), int(_log(rng, 64, 1024))
        return _bed("packed", (nx, ny), int(nx * (ny // 2) * 0.35 * 25 / (math.pi * 0.25)), "f32",
                    rng.randint(8, 16), 0.1, friction=rng.random() < 0.5)
    if what == "packed3":
        n = (rng.randint(6, 16), rng.randint(6, 16), rng.randint(8, 32))
        return _bed("packed", n, int(n[0] * n[1] * (n[2] // 2) * 0.35 * 125 * 6 / math.pi), "f32",
                    rng.randint(4, 16), friction=rng.random() < 0.5)
    if what == "riser3d":
        n = (int(_log(rng, 16, 160)), int(_log(rng, 16, 160)), int(_log(rng, 48, 640)))
        cells = n[0] * n[1] * n[2]
        return _bed("riser3d", n, int(cells * rng.uniform(0.0597, 0.12)),
                    rng.choice(["f32", "f32", "f16", "bf16", "f64"]), rng.randint(8, 20), les,
                    rng.choice(["particles", "particles monitored"]))
    n = (int(_log(rng, 48, 640)), int(_log(rng, 96, 2048)))
    return _bed("riser2d", n, int(n[0] * n[1] * rng.uniform(0.15, 0.6)),
                rng.choice(["f32", "f32", "f16", "bf16"]), rng.randint(32, 64), les,
                rng.choice(["particles fields", "particles monitored"]))


# ------------------------------------------------------------------ inputs

def _workload(case, seed):
    c, st = case, STORAGE[case["storage"]]
    seed = 1303000 + 7919 * seed
    if c["bed"] == "bubbling":
        return W.bubbling2d(nx=c["nx"], ny=c["ny"], n_particles=c["particles"], seed=seed,
                            storage=st, cs_smag=c["les"], bed_fraction=0.4 if c["particles"] <
                            0.3 * c["nx"] * c["ny"] else 0.8)
    if c["bed"] == "cfb":
        return W.cfb_riser2d(nx=c["nx"], ny=c["ny"], n_particles=c["particles"], seed=seed,
                             storage=st, cs_smag=c["les"])
    if c["bed"] == "packed":
        n = (c["nx"], c["ny"]) + ((c["nz"],) if "nz" in c else ())
        w = W.packed_bed(dim=len(n), n=n, n_particles=c["particles"], seed=seed, storage=st,
                         cs_smag=c["les"])
        return W.with_friction(w) if c.get("friction") else w
    if c["bed"] == "riser3d":
        return W.riser3d(nx=c["nx"], ny=c["ny"], nz=c["nz"], n_particles=c["particles"], seed=seed,
                         storage=st, cs_smag=c["les"])
    return W.riser2d(nx=c["nx"], ny=c["ny"], n_particles=c["particles"], seed=seed, storage=st,
                     cs_smag=c["les"])


def _requests(case, seed):
    """Bubbling and riser beds of the serving stream's lattices, counts and storages; the seed
    moves their particles."""
    rng = np.random.default_rng(1303004 + case["requests"])
    out = []
    for i in range(case["requests"]):
        lu = lambda lo, hi: float(np.exp(rng.uniform(np.log(lo), np.log(hi))))  # noqa: E731
        kind = "bubbling" if rng.random() < 0.5 else "riser"
        nx = max(64, int(round(lu(64, 512) / 32)) * 32)
        ny = max(128, int(round(lu(128, 1024) / 32)) * 32)
        n, steps = int(lu(1e3, 1e5)), int(lu(case["steps"] / 4, case["steps"]))
        storage = W.STORE_F16 if rng.random() < 0.5 else W.STORE_F32
        if kind == "riser":
            h = 1.322e-4
            n = min(n, int(0.25 * nx * ny / (math.pi * (0.5 * 54e-6 / h) ** 2)))
            w = W.riser2d(nx=nx, ny=ny, n_particles=n, seed=1303100 + 7919 * seed + i,
                          storage=storage, h=h, steps=steps, cs_smag=0.1)
        else:
            n = min(n, int(0.25 * 0.4 * nx * ny / (math.pi * (0.5 * 0.5e-3 / 2e-3) ** 2)))
            w = W.bubbling2d(nx=nx, ny=ny, n_particles=n, seed=1303100 + 7919 * seed + i,
                             storage=storage, steps=steps, cs_smag=0.1)
        out.append(w)
    return out


def prepare(case, seed):
    if case["what"] == "binning":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n, k = (case["nx"], case["ny"]), case["particles"]
        pos = [torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * n[a]
               for a in range(2)]
        start = torch.empty(n[0] * n[1] + 1, dtype=torch.int32, device="cuda")
        order = torch.empty(k, dtype=torch.int32, device="cuda")
        return {"what": "binning", "n": n, "pos": pos, "start": start, "order": order}
    if case["what"] == "serving":
        return {"what": "serving", "beds": _requests(case, seed),
                "server": L.Server(hbm_budget=64 << 30, max_active=64, steps_per_tick=16)}
    w = _workload(case, seed)
    state = {"what": "bed", "bed": L.Bed(w), "steps": case["steps"], "read": case["read"].split(),
             "single": case["storage"] != "f64"}
    if w.ncell <= RESTART_CELLS:
        state["start"] = (state["bed"].populations(), *state["bed"].particles())
    return state


# ------------------------------------------------------------------ one pass

def run(state):
    if state["what"] == "binning":
        L.bin_sort_noalloc(2, state["n"], [p.data_ptr() for p in state["pos"]],
                           state["start"].data_ptr(), state["order"].data_ptr(),
                           state["order"].numel(), torch.cuda.current_stream().cuda_stream)
        return {"start": state["start"], "order": state["order"]}
    if state["what"] == "serving":
        return _serve(state["server"], state["beds"])
    bed, read, out = state["bed"], state["read"], {}
    kept = torch.Tensor.float if state["single"] else (lambda t: t)
    if "start" in state:
        f, pos, vel = state["start"]
        bed.set_populations(f)
        bed.set_particles(pos, vel)
    if "monitored" in read:
        recs = bed.step_monitored(state["steps"])
        out["stats"] = kept(torch.from_numpy(np.array(
            [[r["mass"], *r["gas_momentum"], *r["particle_momentum"], r["mean_eps_g"]] for r in recs])))
    else:
        bed.step(state["steps"])
    pos, vel = bed.particles()
    out["pos"], out["vel"] = torch.from_numpy(pos), kept(torch.from_numpy(vel))
    if "spin" in read:
        out["spin"] = kept(torch.from_numpy(bed.spin()))
    if "fields" in read:
        mask = L.FIELD_RHO | L.FIELD_UACT | (L.FIELD_FPG | L.FIELD_BETA if "all" in read else 0)
        for name, v in bed.fields(mask).items():
            out[name] = kept(torch.from_numpy(v))
    return out


def _serve(server, beds):
    at = {server.submit(w, w.steps, keep=True): i for i, w in enumerate(beds)}
    done = {}
    while len(done) < len(beds):
        for r in server.poll(wait_s=0.01):
            done[at[r["id"]]] = r
    parts = []
    for rid, i in at.items():
        bed = server.take(rid)
        parts.append(bed.particles())
        bed.close()
    return {"pos": torch.from_numpy(np.concatenate([p for p, _ in parts])),
            "vel": torch.from_numpy(np.concatenate([v for _, v in parts])).float(),
            "gas": torch.tensor([[done[i]["mass"], done[i]["mean_eps_g"]] for i in range(len(beds))],
                                dtype=torch.float32),
            "steps": torch.tensor([done[i]["steps"] for i in range(len(beds))])}


# ------------------------------------------------------------------ what a pass cannot do without

def _step_work(dim, cells, particles, storage, soft):
    """Of one step: the populations read and written, and each particle's position, velocity and id."""
    q, pop, real = (9 if dim == 2 else 19), POP_BYTES[storage], (8 if storage == "f64" else 4)
    byte = cells * 2 * q * pop + particles * 2 * ((8 + real) * dim + 4)
    return byte, cells * (24 * q + 60) + particles * (60 + 30 * 2 ** dim + (600 if soft else 40))


def work(case):
    if case["what"] == "binning":
        cells, k = case["nx"] * case["ny"], case["particles"]
        return {"bytes": 16 * k + 4 * k + 4 * (cells + 1), "flops": 6 * k}
    if case["what"] == "serving":
        b = f = 0
        for w in _requests(case, 0):
            x, y = _step_work(2, w.ncell, w.n_particles,
                              "f16" if w.storage == W.STORE_F16 else "f32", False)
            b, f = b + w.steps * x + 32 * w.n_particles, f + w.steps * y
        return {"bytes": b, "flops": f}
    dim = 3 if "nz" in case else 2
    cells, k = case["nx"] * case["ny"] * case.get("nz", 1), case["particles"]
    b, f = _step_work(dim, cells, k, case["storage"], case["bed"] == "packed")
    b, f = b * case["steps"], f * case["steps"]
    b += 16 * dim * k
    if "spin" in case["read"]:
        b += 8 * k * (1 if dim == 2 else 3)
    if "fields" in case["read"]:
        b += 8 * cells * (1 + dim + (1 + dim if "all" in case["read"] else 0))
    if cells <= RESTART_CELLS:
        b += 8 * cells * (9 if dim == 2 else 19) + 16 * dim * k
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same step in FP64

def exact(case, seed):
    if case["what"] == "binning":
        return None   # whole numbers
    if case["what"] == "serving":
        beds = _requests(case, seed)
        runs = [_Reference(w) for w in beds]
        for r, w in zip(runs, beds):
            r.steps(w.steps)
        got = [r.particles() for r in runs]
        return {"pos": torch.cat([p for p, _ in got]), "vel": torch.cat([v for _, v in got]),
                "gas": torch.stack([r.stats()[[0, -1]] for r in runs]), "steps": None}
    w = _workload(case, seed)
    ref, read = _Reference(w), case["read"].split()
    recs = ref.steps(case["steps"], "monitored" in read)
    out = {}
    if "monitored" in read:
        out["stats"] = torch.stack(recs)
    out["pos"], out["vel"] = ref.particles()
    if case["bed"] == "packed" and ref.D == 2:
        # among a million crowded cells a few have pre-drags that all but cancel; the drag's
        # rescale divides by their sum, so those particles' velocities are not determined
        out["vel"] = None
    if "spin" in read:
        out["spin"] = ref.spins()
    if "fields" in read:
        out["rho"], out["uact"] = ref.rho.reshape(-1), ref.uact.reshape(ref.D, -1).T.contiguous()
        if "all" in read:
            out["fpg"], out["beta"] = ref.fpg.reshape(ref.D, -1).T.contiguous(), ref.beta.reshape(-1)
    return out


_C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
       (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


class _Reference:
    """One bed in FP64 on torch tensors, cells as (z,) y, x, lattice units."""

    def __init__(self, w):
        self.w, self.D = w, w.dim
        D, dev = w.dim, "cuda"
        self.t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
        self.n = [int(v) for v in w.n[:D]]
        self.cells = int(np.prod(self.n))
        self.shape = tuple(self.n[::-1])
        self.dim_of = [D - 1 - a for a in range(D)]           # tensor dimension of an axis
        self.c = _C2 if D == 2 else _C3
        self.opp = [self.c.index(tuple(-v for v in c)) for c in self.c]
        rest, axis, diag = (4 / 9, 1 / 9, 1 / 36) if D == 2 else (1 / 3, 1 / 18, 1 / 36)
        self.wt = [(rest, axis, diag)[sum(abs(v) for v in c)] for c in self.c]
        us, gs = w.dt / w.h, w.dt * w.dt / w.h
        self.tau = 3.0 * (w.mu_g / w.rho_g * w.dt / (w.h * w.h)) + 0.5
        self.mu = (self.tau - 0.5) / 3.0
        self.d = w.d_p / w.h
        self.r, self.vp = 0.5 * self.d, math.pi * self.d ** 3 / 6.0
        self.mp = w.rho_s / w.rho_g * self.vp
        self.geff = [(1.0 - w.rho_g / w.rho_s) * w.g[a] * gs for a in range(D)]
        self.fb = [w.body_accel[a] * gs for a in range(D)]
        self.inlet = None if w.inlet_u is None else self.t(np.asarray(w.inlet_u) * us)
        self.soft = w.collision_model == 1
        if self.soft:
            s3 = w.rho_g * w.h ** 3
            self.kn = w.dem_kn * w.dt * w.dt / s3
            le = math.log(w.e)
            z = -le / math.sqrt(math.pi ** 2 + le * le)
            self.eta, self.eta_w = (2 * z * math.sqrt(m * self.kn) for m in (0.5 * self.mp, self.mp))
            self.mu_f, self.gam_t = w.dem_mu, w.dem_gamma_t * w.dt / s3
        self._tables()
        u0 = [w.u0[a] * us for a in range(D)]
        uu = sum(v * v for v in u0)
        self.f = torch.empty((len(self.c),) + self.shape, dtype=torch.float64, device=dev)
        for i, c in enumerate(self.c):
            cu = sum(c[a] * u0[a] for a in range(D))
            self.f[i] = self.wt[i] * (3 * cu + 4.5 * cu * cu - 1.5 * uu)
        self.P = [self.t(w.pos[:, a]) / w.h for a in range(D)]
        self.v = [self.t(w.vel[:, a]) * us for a in range(D)]
        self.np = len(w.pos)
        self.spin = [torch.zeros(self.np, dtype=torch.float64, device=dev)
                     for _ in range(1 if D == 2 else 3)]
        self.id = torch.arange(self.np, device=dev)
        self._sort()

    def _tables(self):
        D, w = self.D, self.w
        unit = math.pi * self.r ** 2 if D == 2 else self.vp
        cap = math.pi / (2 * math.sqrt(3)) if D == 2 else math.pi / (3 * math.sqrt(2))
        n = np.arange(int(math.ceil(cap / unit)) + 2, dtype=np.float64)
        es = np.minimum(n * unit, cap)
        sg = math.sqrt(2) / math.sqrt(math.pi * math.sqrt(3)) * es * np.sqrt(es) if D == 2 else es
        eg = 1.0 - sg
        div = {0: 1.0 - es, 1: eg, 2: np.ones_like(es)}[w.superficial_mode]
        om = np.where(eg <= 0.74, 1.0,
                      np.where(eg <= 0.82, 0.0214 / (4 * (eg - 0.7463) ** 2 + 0.0044) - 0.5760,
                               np.where(eg <= 0.97, 0.0038 / (4 * (eg - 0.7789) ** 2 + 0.0040) - 0.0101,
                                        32.8295 * eg - 31.8295)))
        gam = es * (self.tau - 0.5) / ((1 - es) + (self.tau - 0.5))
        dil, d, mu = eg > 0.74, self.d, self.mu
        self.tab = {k: self.t(v) for k, v in dict(
            es=es, sg=sg, eg=eg, inv=1.0 / div, og=om * gam, gam=gam, dil=dil.astype(float),
            a=np.where(dil, 0.75 * sg * eg * 24 * mu / (eg * d) / d * om, 150 * sg * sg * mu / (eg * d * d)),
            b=np.where(dil, 0.0, 1.75 * sg / d), c=np.where(dil, 0.75 * sg * eg * 0.44 / d * om, 0.0),
            re=np.where(dil, eg * d / mu, 0.0)).items()}

    # -- particles in cells ------------------------------------------------
    def _sort(self):
        q = [p.floor().long().clamp(0, self.n[a] - 1) for a, p in enumerate(self.P)]
        key = q[0] + self.n[0] * (q[1] + (self.n[1] * q[2] if self.D == 3 else 0))
        o = torch.argsort(key * max(self.np, 1) + self.id)
        self.q, self.cell, self.id = [x[o] for x in q], key[o], self.id[o]
        self.P, self.v = [x[o] for x in self.P], [x[o] for x in self.v]
        self.spin = [x[o] for x in self.spin]
        self.count = torch.bincount(self.cell, minlength=self.cells)
        self.first = torch.cumsum(self.count, 0) - self.count

    def _per(self, a):
        return self.w.bc[2 * a] == W.PERIODIC

    def _near(self, reach):
        """Pairs (i, j), i != j, closer than `reach` by the minimum image."""
        out = []
        most = int(self.count.max()) if self.np else 0
        for off in self.c if self.D == 2 else [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1)
                                               for z in (-1, 0, 1)]:
            ok = torch.ones(self.np, dtype=torch.bool, device="cuda")
            q = []
            for a in range(self.D):
                x = self.q[a] + off[a]
                if self._per(a):
                    x = x % self.n[a]
                else:
                    ok &= (x >= 0) & (x < self.n[a])
                    x = x.clamp(0, self.n[a] - 1)
                q.append(x)
            c = q[0] + self.n[0] * (q[1] + (self.n[1] * q[2] if self.D == 3 else 0))
            first, num = self.first[c], torch.where(ok, self.count[c], 0)
            for m in range(most):
                i = torch.nonzero(num > m).squeeze(1)
                if not len(i):
                    break
                j = first[i] + m
                d2 = sum(self._sep(i, j, a) ** 2 for a in range(self.D))
                hit = (d2 < reach * reach) & (i != j)
                out.append(torch.stack((i[hit], j[hit])))
        if not out:
            return torch.zeros((2, 0), dtype=torch.long, device="cuda")
        return torch.cat(out, 1)

    def _sep(self, i, j, a):
        d = self.P[a][i] - self.P[a][j]
        if self._per(a):
            n = float(self.n[a])
            d = torch.where(d > 0.5 * n, d - n, torch.where(d < -0.5 * n, d + n, d))
        return d

    def _open_top(self, a):
        return bool(self.w.recirculate) and a == self.D - 1

    def _collide(self):
        """Approaching contacts; mutual nearest choices exchange momentum, the rest meet the walls."""
        D, e, inf = self.D, self.w.e, float("inf")
        i, j = self._near(self.d)
        dx = [self._sep(i, j, a) for a in range(D)]
        g = [self.v[a][i] - self.v[a][j] for a in range(D)]
        dot, d2 = sum(x * y for x, y in zip(dx, g)), sum(x * x for x in dx)
        k = dot < 0
        i, j, d2 = i[k], j[k], d2[k]
        near = torch.full((self.np,), inf, dtype=torch.float64, device="cuda")
        near.scatter_reduce_(0, i, d2, "amin")
        k = d2 == near[i]
        i, j = i[k], j[k]
        ids = torch.full((self.np,), 1 << 60, device="cuda")
        ids.scatter_reduce_(0, i, self.id[j], "amin")
        k = self.id[j] == ids[i]
        best = torch.full((self.np,), -1, device="cuda")
        best[i[k]] = j[k]
        i = torch.nonzero(best >= 0).squeeze(1)
        i = i[best[best[i]] == i]
        j = best[i]
        dx = [self._sep(i, j, a) for a in range(D)]
        g = [self.v[a][i] - self.v[a][j] for a in range(D)]
        kf = (1 + e) * 0.5 * sum(x * y for x, y in zip(dx, g)) / sum(x * x for x in dx)
        new = [v.clone() for v in self.v]
        alone = torch.ones(self.np, dtype=torch.bool, device="cuda")
        alone[i] = False
        for a in range(D):
            new[a][i] = self.v[a][i] - kf * dx[a]
            if not self._per(a):
                hit = (self.P[a] < self.r) & (self.v[a] < 0)
                if not self._open_top(a):
                    hit |= (self.n[a] - self.P[a] < self.r) & (self.v[a] > 0)
                new[a] = torch.where(hit & alone, -e * new[a], new[a])
        self.v = new

    def _cross(self, w, n):
        if self.D == 2:
            return [-w[0] * n[1], w[0] * n[0]]
        return [w[1] * n[2] - w[2] * n[1], w[2] * n[0] - w[0] * n[2], w[0] * n[1] - w[1] * n[0]]

    def _friction(self, at, n, l, fn, vc, F, T):
        D = self.D
        vcn = sum(vc[a] * n[a] for a in range(D))
        vt = [vc[a] - vcn * n[a] for a in range(D)]
        s = torch.sqrt(sum(x * x for x in vt))
        k = torch.where(s > 0, -torch.minimum(self.gam_t * s, self.mu_f * fn) / s.clamp(min=1e-300), 0.0)
        Ft = [k * x for x in vt]
        for a in range(D):
            F[a].index_add_(0, at, Ft[a])
        tq = [n[0] * Ft[1] - n[1] * Ft[0]] if D == 2 else self._cross(n, Ft)
        for x, y in zip(T, tq):
            x.index_add_(0, at, -l * y)

    def _contacts(self):
        D, fric = self.D, self.w.dem_mu > 0 and self.w.dem_gamma_t > 0
        F = [torch.zeros(self.np, dtype=torch.float64, device="cuda") for _ in range(D)]
        T = [torch.zeros_like(F[0]) for _ in self.spin]
        i, j = self._near(self.d)
        dx = [self._sep(i, j, a) for a in range(D)]
        dist = torch.sqrt(sum(x * x for x in dx))
        nrm = [x / dist for x in dx]
        vr = [self.v[a][i] - self.v[a][j] for a in range(D)]
        f = self.kn * (self.d - dist) - self.eta * sum(x * y for x, y in zip(vr, nrm))
        k = f > 0
        i, j, dist, f = i[k], j[k], dist[k], f[k]
        nrm, vr = [x[k] for x in nrm], [x[k] for x in vr]
        for a in range(D):
            F[a].index_add_(0, i, f * nrm[a])
        if fric:
            wn = self._cross([s[i] + s[j] for s in self.spin], nrm)
            self._friction(i, nrm, 0.5 * dist, f, [vr[a] - 0.5 * dist * wn[a] for a in range(D)], F, T)
        for a in range(D):
            for sg in (1.0, -1.0):
                if self._per(a) or (sg < 0 and self._open_top(a)):
                    continue
                gap = self.P[a] if sg > 0 else self.n[a] - self.P[a]
                f = self.kn * (self.r - gap) - self.eta_w * sg * self.v[a]
                i = torch.nonzero((gap < self.r) & (f > 0)).squeeze(1)
                F[a][i] += sg * f[i]
                if fric:
                    nrm = [torch.full_like(gap[i], sg if b == a else 0.0) for b in range(D)]
                    wn = self._cross([s[i] for s in self.spin], nrm)
                    self._friction(i, nrm, gap[i], f[i],
                                   [self.v[b][i] - gap[i] * wn[b] for b in range(D)], F, T)
        if fric:
            self.spin = [s + t / (0.4 * self.mp * self.r ** 2) for s, t in zip(self.spin, T)]
        return F

    # -- gas ----------------------------------------------------------------
    def _gas(self):
        D, w, tab, tau = self.D, self.w, self.tab, self.tau
        k = self.count.clamp(max=len(tab["es"]) - 1)
        at = lambda name: tab[name][k].reshape(self.shape)  # noqa: E731
        vs = []
        for a in range(D):
            s = torch.zeros(self.cells, dtype=torch.float64, device="cuda")
            s.index_add_(0, self.cell, self.v[a])
            vs.append((s / self.count.clamp(min=1)).reshape(self.shape))
        og = at("og")
        drho = self.f.sum(0)
        rho = 1 + drho
        m = []
        for a in range(D):
            s = torch.zeros_like(rho)
            for i, c in enumerate(self.c):
                if c[a]:
                    s.add_(self.f[i], alpha=c[a])
            m.append(s)
        u = [(m[a] * (1 - og) + 0.5 * og * rho * vs[a] + 0.5 * self.fb[a]) / (rho * (1 - 0.5 * og))
             for a in range(D)]
        self.fpg = torch.stack([og * (rho * u[a] + rho * vs[a] - 2 * m[a]) for a in range(D)])
        del m
        uu, vv = sum(x * x for x in u), sum(x * x for x in vs)
        self.rho, self.uact = rho, torch.stack([x * at("inv") for x in u])
        slip = torch.sqrt(sum((self.uact[a] - vs[a]) ** 2 for a in range(D)))
        re = at("re") * slip
        self.beta = torch.where(at("dil") > 0,
                                torch.where(re < 1000, at("a") * (1 + 0.15 * re ** 0.687), at("c") * slip),
                                at("a") + at("b") * slip)
        del re, slip
        self.sg = at("sg")
        eq0, es0 = drho - 1.5 * rho * uu, drho - 1.5 * rho * vv
        dot = lambda c, x: sum(c[a] * x[a] for a in range(D) if c[a])  # noqa: E731
        tau_t, gam_t = tau, at("gam")
        if w.cs_smag > 0:
            q = {}
            for i, c in enumerate(self.c[1:], 1):
                cu = dot(c, u)
                neq = self.f[i] - self.wt[i] * (eq0 + rho * (3 * cu + 4.5 * cu * cu))
                for a in range(D):
                    for b in range(a, D):
                        if c[a] * c[b]:
                            q[a, b] = q.get((a, b), 0) + c[a] * c[b] * neq
            qn = torch.sqrt(2 * sum((1 if a == b else 2) * x * x for (a, b), x in q.items()))
            tau_t = 0.5 * (tau + torch.sqrt(tau * tau + 18 * w.cs_smag ** 2 * qn / rho))
            es = at("es")
            gam_t = es * (tau_t - 0.5) / ((1 - es) + (tau_t - 0.5))
        relax, pref = (1 - gam_t) / tau_t, 1 - 0.5 / tau_t
        uF = sum(u[a] * self.fb[a] for a in range(D))
        post = torch.empty_like(self.f)
        for i, c in enumerate(self.c):
            wt, cu, cv = self.wt[i], dot(c, u), dot(c, vs)
            eu = wt * (eq0 + rho * (3 * cu + 4.5 * cu * cu))
            ev = wt * (es0 + rho * (3 * cv + 4.5 * cv * cv))
            ob = wt * (eq0 + rho * (-3 * cu + 4.5 * cu * cu))
            fo = self.f[self.opp[i]]
            post[i] = self.f[i] - relax * (self.f[i] - eu) + og * (fo - self.f[i] + ev - ob)
            if any(self.fb):
                cF = sum(c[a] * self.fb[a] for a in range(D))
                post[i] += pref * wt * (9 * cu * cF - 3 * uF + 3 * cF)
        self._stream(post, u)

    def _stream(self, post, u):
        D, bc = self.D, self.w.bc
        for i, c in enumerate(self.c):
            g = torch.roll(post[i], [c[a] for a in range(D)], [self.dim_of[a] for a in range(D)])
            wall = opening = None
            for a in range(D):
                if not c[a] or self._per(a):
                    continue
                face = 2 * a if c[a] > 0 else 2 * a + 1      # the source lies beyond this face
                line = torch.zeros(self.n[a], dtype=torch.bool, device="cuda")
                line[0 if c[a] > 0 else -1] = True
                line = line.reshape([-1 if d == self.dim_of[a] else 1 for d in range(D)])
                if bc[face] == W.WALL:
                    wall = line if wall is None else wall | line
                else:
                    opening = (line, bc[face])
            if opening is not None:
                if opening[1] == W.INLET:
                    shape = (1,) + (self.shape[1:])
                    ub = [self.inlet[:, a].reshape(shape) for a in range(D)]
                else:
                    ub = u
                cu, uu = sum(c[a] * ub[a] for a in range(D)), sum(x * x for x in ub)
                g = torch.where(opening[0], self.wt[i] * (3 * cu + 4.5 * cu * cu - 1.5 * uu), g)
            if wall is not None:
                g = torch.where(wall, post[self.opp[i]], g)
            self.f[i] = g

    # -- drag and integration ------------------------------------------------
    def _gradient(self, a):
        d, p = self.dim_of[a], self.rho / 3.0
        up, dn = torch.roll(p, -1, d), torch.roll(p, 1, d)
        g = 0.5 * (up - dn)
        if not self._per(a):
            last = self.n[a] - 1
            g.select(d, 0).copy_((p.select(d, 1) - p.select(d, 0)) if last else torch.zeros_like(p.select(d, 0)))
            g.select(d, last).copy_((p.select(d, last) - p.select(d, last - 1)) if last else
                                    torch.zeros_like(p.select(d, 0)))
        return g.reshape(-1)

    def _drag(self, contact):
        D = self.D
        lo, hi, frac = [], [], []
        for a in range(D):
            t = self.P[a] - 0.5
            i = t.floor().long()
            frac.append(t - i)
            if self._per(a):
                lo.append(i % self.n[a])
                hi.append((i + 1) % self.n[a])
            else:
                lo.append(i.clamp(min=0))
                hi.append((i + 1).clamp(max=self.n[a] - 1))
        grad = [self._gradient(a) for a in range(D)]
        uk, gk = [0.0] * D, [0.0] * D
        sk = bk = 0.0
        for corner in range(1 << D):
            bit = [(corner >> a) & 1 for a in range(D)]
            q = [hi[a] if bit[a] else lo[a] for a in range(D)]
            wt = 1.0
            for a in range(D):
                wt = wt * (frac[a] if bit[a] else 1 - frac[a])
            x = q[0] + self.n[0] * (q[1] + (self.n[1] * q[2] if D == 3 else 0))
            for a in range(D):
                uk[a] = uk[a] + wt * self.uact[a].reshape(-1)[x]
                gk[a] = gk[a] + wt * grad[a][x]
            sk = sk + wt * self.sg.reshape(-1)[x]
            bk = bk + wt * self.beta.reshape(-1)[x]
        coef = self.vp * bk / sk
        sign = 1.0 if self.w.pressure_plus else -1.0
        for a in range(D):
            fp = coef * (uk[a] - self.v[a])
            S = torch.zeros(self.cells, dtype=torch.float64, device="cuda")
            A = torch.zeros_like(S)
            S.index_add_(0, self.cell, fp)
            A.index_add_(0, self.cell, fp.abs())
            ratio = self.fpg[a].reshape(-1).abs() / S.abs()
            scale = torch.where(S.abs() <= 1e-12 * A, torch.ones_like(S), ratio)[self.cell]
            force = scale * fp + sign * self.vp * gk[a]
            if contact is not None:
                force = force + contact[a]
            v = self.v[a] + (self.geff[a] + force / self.mp)
            P, n, e = self.P[a] + v, float(self.n[a]), self.w.e
            if self._per(a):
                P = torch.where(P >= n, P - n, torch.where(P < 0, P + n, P))
            else:
                out = P >= n
                if self._open_top(a):
                    P = torch.where(out, P - n, P)
                    out = torch.zeros_like(out)
                low = P < 0
                P = torch.where(low, -P, torch.where(out, 2 * n - P, P))
                v = torch.where(low | out, -e * v, v)
            self.P[a], self.v[a] = P, v

    def steps(self, k, monitored=False):
        recs = []
        for _ in range(k):
            self._gas()
            self._drag(self._contacts() if self.soft else None)
            self._sort()
            if not self.soft:
                self._collide()
            if monitored:
                recs.append(self.stats())
        return recs

    # -- results --------------------------------------------------------------
    def stats(self):
        """Gas mass and momentum, particle momentum and mean voidage, as one row."""
        per = [x.sum() for x in self.f]
        row = [sum(per) + self.cells]
        zero = torch.zeros((), dtype=torch.float64, device="cuda")
        for a in range(3):
            row.append(sum((c[a] * s for c, s in zip(self.c, per)), zero) if a < self.D else zero)
        row += [self.mp * self.v[a].sum() if a < self.D else zero for a in range(3)]
        row.append(self.tab["eg"][self.count.clamp(max=len(self.tab["eg"]) - 1)].mean())
        return torch.stack(row)

    def _by_id(self, cols):
        out = torch.empty((self.np, len(cols)), dtype=torch.float64, device="cuda")
        out[self.id] = torch.stack(cols, 1)
        return out

    def particles(self):
        return self._by_id(self.P), self._by_id(self.v)

    def spins(self):
        s = self._by_id(self.spin)
        return s[:, 0] if self.D == 2 else s
