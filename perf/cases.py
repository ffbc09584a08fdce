"""Performance cases of the library: what its users have it do, each through the public entry points.

A case is a plain dict.  `prepare` builds what a program holds before the call (a handle with its sphere, parameters and
seeded initial flow), `run` takes one pass (some time steps and the read-back of the particle, or one gradient of the
mean drag) and returns the whole result: the population fields, the particle's record or history, J and its gradients.

The population fields stay on the device.  The program hands the library its own device memory through the allocator
of lbmp_config (as the C ABI offers it), so it can look at a field where it lies:
  uniform grid   the two allocations of a field's size are its two copies, [q][z][y][x] in the storage type (FP16: the
                 deviation times 2^fp16_scale_log2); a step reads one and writes the other, so after k steps the field
                 is in copy k mod 2 (in the order of the allocations);
  batched        the same two copies for all simulations, one after another;
  refined grid   two pools of equal size per level, levels in order, [block][q][16^3 cells], real blocks first, in the
                 order of lbmp_get_block_map; after an even number of level-0 steps the fields are in the first ones.
Records that the C ABI widens to FP64 come back in the type the simulation computes in.

`exact` is the method of the paper (arXiv 2103.10882) written out in plain torch, in 64 bits, for the uniform, batched
and differentiated cases.
"""
import ctypes
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_2103_10882_gb300 as L
from paper_2103_10882_gb300 import workloads

MAGIC = 3.0 / 16.0
U_G = 0.01            # the paper's gravitational velocity
ESIZE = {"fp64": 8, "fp32": 4, "fp16": 2}
DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16}
RECORD = {"fp64": np.float64, "fp32": np.float32, "fp16": np.float32}
FP16_SCALE = 11
CELL_STEPS = 5.4e8    # cell updates of the largest listed case (512^3, four steps)


# ------------------------------------------------------------------ the cases
def _uniform(name, shape, d, steps, precision="fp32", tau=0.0, ga=0.0, pi=0.5, cv=0.5, walls=0, wall_u=0.0, bulk=1.0,
             refill="equilibrium", held="", amplitude=1e-3, read="history"):
    """tau > 0 sets the relaxation time, else it follows from the Galileo number.  walls: 1 no-slip on z, 2 on x and y."""
    return dict(name=name, kind="uniform", nx=shape[0], ny=shape[1], nz=shape[2], diameter=float(d), steps=steps,
                precision=precision, tau=float(tau), ga=float(ga), density_ratio=float(pi), cv=float(cv), walls=walls,
                wall_u=float(wall_u), bulk=float(bulk), refill=refill, held=held, amplitude=float(amplitude), read=read)


def _refined(name, shape, levels, d, steps, precision="fp32", tau=0.0, ga=0.0, pi=0.5, cv=0.5, walls=0, interval=50,
             sensor=True, amplitude=0.0):
    return dict(name=name, kind="refined", nx=shape[0], ny=shape[1], nz=shape[2], levels=levels, diameter=float(d),
                steps=steps, precision=precision, tau=float(tau), ga=float(ga), density_ratio=float(pi), cv=float(cv),
                walls=walls, interval=interval, sensor=sensor, amplitude=float(amplitude))


def _batch(name, count, steps, sweep, precision="fp32", largest=96):
    return dict(name=name, kind="batch", count=count, steps=steps, sweep=sweep, precision=precision, largest=largest)


def _drag(name, shape, d, steps, checkpoint_every, precision="fp32", tau=0.6, force=1e-6, axis=0):
    return dict(name=name, kind="drag", nx=shape[0], ny=shape[1], nz=shape[2], diameter=float(d), steps=steps,
                checkpoint_every=checkpoint_every, precision=precision, tau=float(tau), force=float(force), axis=axis)


def listed():
    w = workloads.SINGLE_SPHERE_32
    a = workloads.ADJOINT_64
    r = workloads.ROOFLINE_512
    return [
        # the smallest call: a program that steers or records every step (set gravity, one step, read the particle)
        _uniform("sphere32_each_step", w["shape"], w["diameter"], 1, tau=w["tau"], read="particle"),
        # the single-sphere run, read back every 100 steps: a short test or a parameter scan on a small box
        _uniform("sphere32_run", w["shape"], w["diameter"], 100, tau=w["tau"]),
        # a stability-limit run (Sec. 3.2): (6.4, 6.4, 12.8) d_p periodic box, the paper's collision with Lambda_b = 100
        _uniform("stability_d10_mrt", (64, 64, 128), 10, 50, ga=100, bulk=100, amplitude=0),
        # the rotating virtual-mass test (Sec. 3.4) at d_p = 20: moving upper wall, translation held
        _uniform("rotation_d20_walls", (256, 128, 96), 20, 50, tau=0.5 + 3.0 * 0.05 * 20 / 110, pi=0.1, walls=1,
                 wall_u=0.1, held="translation"),
        # FP16 storage on a field far larger than the L2: the mode for large fields
        _uniform("box256_fp16", (256, 256, 256), 40, 20, "fp16", ga=200),
        # a validation run in FP64 on odd extents, walls in x and y, with the paper's Grad refill
        _uniform("ragged_fp64_grad", (61, 53, 75), 12, 20, "fp64", tau=0.6, walls=2, refill="grad"),
        # the bandwidth case: the largest field of one GPU's work
        _uniform("box512", r["shape"], r["diameter"], 4, ga=r["ga"]),
        # a small refined run in FP64: two levels, a few level-0 steps, regrids among them
        _refined("refined_small_fp64", (32, 32, 48), 2, 8, 10, "fp64", tau=0.6, interval=4, amplitude=1e-3),
        # the refined rising sphere (the headline workload): three levels, walls, regrids with the curl sensor
        _refined("refined_rising", (64, 64, 256), 3, 20, 50, ga=200, walls=2),
        # the batched (density ratio, Ga) sweep: 64 uneven boxes advanced together
        _batch("batch64", 64, 20, 0),
        # a small gradient of the mean drag in FP64 (a gradient check, or an optimisation on a coarse box)
        _drag("drag24_fp64", (24, 24, 24), 6, 30, 7, "fp64", tau=0.7, force=1e-5),
        # the differentiation workload: 64^3, 500 steps, checkpoints every 50, forward and backward
        _drag("drag64", a["shape"], a["diameter"], a["steps"], a["checkpoint"], tau=a["tau"], force=a["body_force"]),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(["uniform", "refined", "batch", "drag"], [5, 3, 2, 3])[0]
    if kind == "uniform":
        precision = rng.choices(["fp32", "fp16", "fp64"], [6, 2, 2])[0]
        edge = _log(rng, 26, 300 if precision != "fp64" else 160)
        f = [_log(rng, 0.7, 1.5) for _ in range(3)]
        shape = [max(24, int(round(edge * v))) for v in f]
        if rng.random() < 0.5:     # whole multiples of 8, as round diameters give them
            shape = [max(24, 8 * (v // 8)) for v in shape]
        d = round(_log(rng, 5.0, min(48.0, 0.28 * min(shape))), 1)
        walls = rng.choices([0, 1, 2], [4, 2, 1])[0]
        n = shape[0] * shape[1] * shape[2]
        steps = max(1, min(rng.choice([1, 10, 50, 100]), int(0.5 * CELL_STEPS / n)))
        c = _uniform("", shape, d, steps, precision, tau=0.5 + _log(rng, 0.02, 0.4), pi=_log(rng, 0.1, 2.5), walls=walls,
                     wall_u=rng.choice([0.0, 0.05]) if walls == 1 else 0.0, bulk=rng.choice([1.0, 1.0, 100.0]),
                     refill=rng.choice(["equilibrium", "equilibrium", "grad"]),
                     held="translation" if walls == 1 else rng.choice(["", "", "", "translation"]),   # walls in its way
                     read="particle" if steps == 1 else "history")
        if abs(c["density_ratio"] - 1.0) < 0.05:
            c["density_ratio"] = 0.9
    elif kind == "refined":
        levels = rng.choice([2, 2, 3])
        shape = [16 * rng.randint(2, 4), 16 * rng.randint(2, 4), 16 * rng.randint(2, 8)]
        walls = rng.choice([0, 2])
        c = _refined("", shape, levels, round(_log(rng, 6.0, 24.0), 1), 2 * rng.randint(1, 15),
                     rng.choices(["fp32", "fp16", "fp64"], [5, 3, 2])[0], tau=0.5 + _log(rng, 0.04, 0.3),
                     pi=_log(rng, 0.1, 0.9), walls=walls, interval=2 * rng.randint(2, 25), sensor=rng.random() < 0.5,
                     amplitude=rng.choice([0.0, 1e-3]))
    elif kind == "batch":
        c = _batch("", int(round(_log(rng, 1, 48))), 2 * rng.randint(1, 10), rng.randint(1, 10 ** 6),
                   rng.choices(["fp32", "fp16", "fp64"], [6, 2, 1])[0], rng.choice([48, 64, 96]))
    else:
        shape = [int(round(_log(rng, 16, 72))) for _ in range(3)]
        n = shape[0] * shape[1] * shape[2]
        steps = max(4, min(int(round(_log(rng, 8, 300))), int(1.2e8 / n)))
        c = _drag("", shape, round(rng.uniform(4.0, 0.4 * min(shape)), 1), steps, max(1, int(round(_log(rng, 4, 50)))),
                  rng.choices(["fp32", "fp64"], [3, 1])[0], tau=0.5 + _log(rng, 0.05, 0.4), force=_log(rng, 1e-6, 1e-5),
                  axis=rng.randint(0, 2))
    del c["name"]
    return c


# ------------------------------------------------------- seeded inputs of a case
def _tau_gravity(c):
    """(tau, |g|) from the case's tau or Galileo number at u_g = 0.01."""
    g = U_G ** 2 / (abs(c["density_ratio"] - 1.0) * c["diameter"])
    return (c["tau"] if c["tau"] > 0 else 0.5 + 3.0 * U_G * c["diameter"] / c["ga"]), g


def _flow(shape, amplitude, seed, walls, wall_u):
    """Seeded divergence-free velocity (3, nz, ny, nx) of six Fourier modes, largest component sum about `amplitude`,
    on top of the Couette profile of a moving upper wall; None for fluid at rest."""
    if amplitude == 0 and wall_u == 0:
        return None
    nx, ny, nz = shape
    dev = "cuda"
    u = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device=dev)
    rs = np.random.RandomState(seed % (1 << 31))
    for _ in range(6 if amplitude else 0):
        k = rs.randint(-2, 3, size=3)
        k[rs.randint(3)] = 1 + rs.randint(2)
        a = rs.uniform(-1, 1, size=(2, 3))
        kv = k / np.array(shape, dtype=np.float64)
        a = a - (a @ kv)[:, None] * kv / (kv @ kv)          # normal to the wave vector
        ph = [torch.polar(torch.ones(n, dtype=torch.float64, device=dev),
                          2.0 * math.pi * int(kk) * (torch.arange(n, dtype=torch.float64, device=dev) + 0.5) / n)
              for kk, n in zip(k, shape)]
        wave = ph[2][:, None, None] * (ph[1][:, None] * ph[0])
        for i in range(3):
            u[i] += (amplitude / 6.0) * (a[0, i] * wave.real + a[1, i] * wave.imag)
    if walls == 1:
        u[0] += (wall_u * (torch.arange(nz, dtype=torch.float64, device=dev) + 0.5) / nz)[:, None, None]
    return u


def _start(c, seed):
    """Sphere centre: the middle of the box plus a seeded sub-cell offset."""
    f = 1 << (c.get("levels", 1) - 1)
    off = workloads.sub_cell_offset(seed)
    return tuple(0.5 * f * c[n] + o for n, o in zip(("nx", "ny", "nz"), off))


def _sweep(c, seed):
    """The simulations of a batched case: the sweep's boxes, with sub-cell offsets from the seed."""
    sims = []
    for i, d in enumerate(workloads.batch_sweep(c["sweep"], c["count"])):
        e, dia = min(d["edge"], c["largest"]), d["diameter"]
        if e < d["edge"]:
            dia = float(round(e / 6.0))
        g = U_G ** 2 / (abs(d["density_ratio"] - 1.0) * dia)
        off = workloads.sub_cell_offset(seed * 1000 + i)
        sims.append(dict(edge=e, pos=tuple(0.5 * e + o for o in off), diameter=dia, density_ratio=d["density_ratio"],
                         cv=0.5, tau=0.5 + 3.0 * U_G * dia / d["ga"], gravity=(0.0, 0.0, -g)))
    return sims


# -------------------------------------------------------------- prepare and run
class _Memory:
    """The program's own device memory behind lbmp_config.alloc: torch buffers, kept in the order they were asked for."""

    def __init__(self, cfg):
        self.live = {}
        self.changes = 0
        self.alloc = type(cfg.alloc)(self._alloc)
        self.free = type(cfg.free)(self._free)
        cfg.alloc, cfg.free = self.alloc, self.free

    def _alloc(self, nbytes, _ctx):
        try:
            t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        except RuntimeError:
            return None
        self.live[t.data_ptr()] = t
        self.changes += 1
        return t.data_ptr()

    def _free(self, ptr, _nbytes, _ctx):
        self.live.pop(ptr, None)
        self.changes += 1

    def copies(self, cells, precision):
        """The two copies of a field of `cells` cells."""
        size = 19 * cells * ESIZE[precision]
        return [t.view(DTYPE[precision]) for t in self.live.values() if t.numel() == size][:2]


class _Handle:
    def __init__(self, cfg, make):
        cfg.cuda_stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        self.memory = _Memory(cfg)
        self.h = make(cfg)

    def __del__(self):
        if getattr(self, "h", None):
            L.lbmp_destroy(self.h)
            self.h = None


def _config(c):
    cfg = L.lbmp_config_default()
    cfg.precision = L.PRECISIONS[c["precision"]]
    cfg.magic = MAGIC
    cfg.fp16_scale_log2 = FP16_SCALE
    cfg.history_capacity = max(64, c["steps"] << (c.get("levels", 1) - 1))   # a record per finest step
    return cfg


def _bc(walls):
    p, w = 0, 1
    return ((p, p, p), (p, p, w), (w, w, p))[walls]


def prepare(case, seed):
    c = case
    kind, prec = c["kind"], c["precision"]
    if kind == "batch":
        cfg = _config(c)
        cfg.history_capacity = 64
        sims = _sweep(c, seed)
        H = _Handle(cfg, lambda k: L.lbmp_batch_create(k, sims))
        L.lbmp_batch_autotune(H.h, 5)
        n = sum(s["edge"] ** 3 for s in sims)
        return dict(case=c, H=H, done=0, count=len(sims), fields=H.memory.copies(n, prec))
    if kind == "drag":
        sim = L.Simulation((c["nx"], c["ny"], c["nz"]), precision=prec, tau=c["tau"])
        sim.add_sphere(_start(c, seed), c["diameter"], 1.0)
        sim.set_fixed(True)
        u0 = _flow(sim.shape, workloads.ADJOINT_64["amplitude"], seed, 0, 0.0).to(DTYPE[prec]).requires_grad_()
        force = [0.0, 0.0, 0.0]
        force[c["axis"]] = c["force"]
        return dict(case=c, sim=sim, u0=u0, tau=torch.tensor(c["tau"], dtype=DTYPE[prec], requires_grad=True),
                    force=torch.tensor(force, dtype=DTYPE[prec], requires_grad=True))
    tau, g = _tau_gravity(c)
    cfg = _config(c)
    cfg.nx, cfg.ny, cfg.nz = c["nx"], c["ny"], c["nz"]
    cfg.tau = tau
    for a, b in enumerate(_bc(c["walls"])):
        cfg.bc[a] = b
    if kind == "uniform":
        cfg.bulk_factor = c["bulk"]
        cfg.refill = L.REFILL[c["refill"]]
        H = _Handle(cfg, L.lbmp_create)
        L.lbmp_add_sphere(H.h, _start(c, seed), c["diameter"], c["density_ratio"], c["cv"])
        L.lbmp_set_gravity(H.h, (0.0, 0.0, -g))
        if c["held"]:
            L.lbmp_set_particle_fixed(H.h, 0, c["held"])
        if c["wall_u"]:
            L.lbmp_set_wall_velocity(H.h, 2, 1, (c["wall_u"], 0.0, 0.0))
        L.lbmp_init_fluid(H.h, u_field=_flow((c["nx"], c["ny"], c["nz"]), c["amplitude"], seed, c["walls"], c["wall_u"]))
        n = c["nx"] * c["ny"] * c["nz"]
        fields = [t.view(19, c["nz"], c["ny"], c["nx"]) for t in H.memory.copies(n, prec)]
        return dict(case=c, H=H, done=0, gravity=(0.0, 0.0, -g), fields=fields)
    cfg.levels = c["levels"]
    cfg.regrid_interval = c["interval"]
    H = _Handle(cfg, L.lbmp_create)
    L.lbmp_add_sphere(H.h, _start(c, seed), c["diameter"], c["density_ratio"], c["cv"])
    L.lbmp_set_gravity(H.h, (0.0, 0.0, -g))
    if c["sensor"]:
        L.lbmp_set_refinement_sensor(H.h, 1e-3, 0.2)
    theta = 2.0 * math.pi * float(workloads.uniform01(seed + 1000, 1)[0])
    L.lbmp_set_particle_velocity(H.h, 0, (1e-3 * U_G * math.cos(theta), 1e-3 * U_G * math.sin(theta), 0.0))
    L.lbmp_init_fluid_wave(H.h, amp=c["amplitude"], direction=0, axis=2)
    return dict(case=c, H=H, seen=-1, fields=None)


def _level_fields(state):
    """Views of every level's real blocks in the program's memory (looked up again after a regrid moved them)."""
    H, c = state["H"], state["case"]
    if state["seen"] != H.memory.changes:
        es = ESIZE[c["precision"]]
        unit = 19 * 4096 * es
        live = list(H.memory.live.values())
        fields, i = [], 0
        for l in range(c["levels"]):
            need = int((L.lbmp_get_block_map(H.h, l) >= 0).sum()) * unit
            while not (live[i].numel() == live[i + 1].numel() and live[i].numel() % unit == 0 and live[i].numel() >= max(need, unit)):
                i += 1
            fields.append(live[i][:need].view(DTYPE[c["precision"]]))
            i += 2
        state["fields"], state["seen"] = fields, H.memory.changes
    return {"level%d" % l: f for l, f in enumerate(state["fields"])}


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "drag":
        tau, force, u0 = state["tau"], state["force"], state["u0"]
        J = L.mean_drag(state["sim"], tau, force, u0, c["steps"], c["checkpoint_every"], c["axis"])
        gt, gf, gu = torch.autograd.grad(J, (tau, force, u0))
        return {"J": J.detach().to(u0.dtype), "grad_tau": gt, "grad_force": gf, "grad_u0": gu}
    h = state["H"].h
    rec = RECORD[c["precision"]]
    if kind == "refined":
        L.lbmp_step(h, c["steps"])
        out = _level_fields(state)
        out["history"] = L.lbmp_get_history(h, 0, c["steps"] << (c["levels"] - 1)).astype(rec)
        return out
    if kind == "uniform" and c["read"] == "particle":
        L.lbmp_set_gravity(h, state["gravity"])
    L.lbmp_step(h, c["steps"])
    state["done"] += c["steps"]
    out = {"field": state["fields"][state["done"] & 1]}
    if kind == "batch":
        out["particles"] = np.stack([L.lbmp_get_particle(h, i) for i in range(state["count"])]).astype(rec)
    elif c["read"] == "particle":
        out["particle"] = L.lbmp_get_particle(h, 0).astype(rec)
    else:
        out["history"] = L.lbmp_get_history(h, 0, c["steps"]).astype(rec)
    return out


# ------------------------------------------------------------------------ work
def work(case):
    """Every cell update reads 19 populations and writes 19; about 190 operations collide them.  The reverse step reads
    the 19 populations and 19 adjoint values and writes 19; a gradient also takes every step once more from its
    checkpoint, which is counted because the fields of all steps cannot be kept."""
    c = case
    es = ESIZE[c["precision"]]
    if c["kind"] == "batch":
        n = sum(s["edge"] ** 3 for s in _sweep(c, 0)) * c["steps"]
    elif c["kind"] == "refined":
        # cell updates of one level-0 step at the start: the sphere's finest blocks with their neighbours, and level 0
        f = 1 << (c["levels"] - 1)
        fine = (2 * math.ceil((c["diameter"] + 2.0) / 32.0) + 2) ** 3 * 4096
        n = (c["nx"] * c["ny"] * c["nz"] + fine * f * (1.5 if c["levels"] > 2 else 1.0)) * c["steps"]
    else:
        n = c["nx"] * c["ny"] * c["nz"] * c["steps"]
    if c["kind"] == "drag":
        return {"bytes": n * es * (2 * 38 + 57), "flops": n * (2 * 190 + 450)}
    return {"bytes": n * es * 38, "flops": n * 190}


# ------------------------------------------- the method in plain torch, 64 bits
C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
     (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
OPP = [0] + [q + 1 if q % 2 else q - 1 for q in range(1, 19)]


def _dot(c, u):
    """sum_a c_a u_a for a lattice velocity (0 where c is the rest velocity)."""
    t = 0.0
    for ca, ua in zip(c, u):
        if ca:
            t = t + ua if ca > 0 else t - ua
    return t


class _Method:
    """One sphere in a uniform box (Sec. 2 and 3 of the paper).  g: deviations f - w, [19, nz, ny, nx] in 64 bits; tau
    and force may be tensors that autograd follows (held sphere at rest only)."""

    def __init__(self, shape, tau, walls=0, wall_u=0.0, bulk=1.0, grad_refill=False, force=None):
        self.n = tuple(shape)
        self.per = [b == 0 for b in _bc(walls)]
        self.wall_u, self.bulk, self.grad_refill = wall_u, bulk, grad_refill
        self.tau, self.force = tau, force
        self.dev = torch.device("cuda")

    def sphere(self, pos, d, pi, cv, gravity, held):
        self.x, self.u, self.w = np.array(pos, dtype=np.float64), np.zeros(3), np.zeros(3)
        self.a, self.b, self.F_old, self.T_old = np.zeros(3), np.zeros(3), None, None
        self.r, self.pi, self.cv, self.V = 0.5 * d, pi, cv, math.pi * d ** 3 / 6.0
        self.gz, self.held = np.array(gravity), held
        self.history, self.Fp = [], np.zeros(3)
        self.flags = self.solid()
        self.links()

    def offsets(self):
        out = []
        for a in range(3):
            d = torch.arange(self.n[a], dtype=torch.float64, device=self.dev) + 0.5 - float(self.x[a])
            if self.per[a]:
                half = 0.5 * self.n[a]
                d = torch.where(d > half, d - self.n[a], torch.where(d < -half, d + self.n[a], d))
            out.append(d)
        return out

    def solid(self):
        dx, dy, dz = (d * d for d in self.offsets())
        return (dx[None, None, :] + dy[None, :, None]) + dz[:, None, None] <= self.r * self.r

    def at(self, cells, c):
        """Neighbours of cells [m, 3] (x, y, z) displaced by c: (linear index, inside)."""
        v = cells + torch.tensor(c, device=self.dev)
        n = torch.tensor(self.n, device=self.dev)
        ok = torch.ones(len(v), dtype=torch.bool, device=self.dev)
        for a in range(3):
            if not self.per[a]:
                ok &= (v[:, a] >= 0) & (v[:, a] < self.n[a])
        v = torch.remainder(v, n)
        return v[:, 0] + self.n[0] * (v[:, 1] + self.n[1] * v[:, 2]), ok

    def box_cells(self, mask):
        """(x, y, z) of the marked cells."""
        z, y, x = torch.nonzero(mask, as_tuple=True)
        return torch.stack((x, y, z), dim=1)

    def links(self):
        """Links (cell, q) whose pull along c_q starts in the sphere, with the wall distance of the opposite direction."""
        near = torch.zeros_like(self.flags)
        for q in range(1, 19):
            cx, cy, cz = C[q]
            near |= torch.roll(self.flags, (cz, cy, cx), (0, 1, 2))
        cells = self.box_cells(near & ~self.flags)
        flat = self.flags.reshape(-1)
        off = self.offsets()
        self.link = []
        for q in range(1, 19):
            s, ok = self.at(cells, tuple(-v for v in C[q]))
            m = ok & flat[s]
            if not bool(m.any()):
                continue
            cl = cells[m]
            far, fok = self.at(cl, C[q])
            fok = fok & ~flat[far]
            x = cl[:, 0] + self.n[0] * (cl[:, 1] + self.n[1] * cl[:, 2])
            d = torch.stack([off[a][cl[:, a]] for a in range(3)], dim=1)
            ck = torch.tensor(C[OPP[q]], dtype=torch.float64, device=self.dev)
            cc, dc = float(ck @ ck), d @ ck
            disc = (dc * dc - cc * ((d * d).sum(1) - self.r * self.r)).clamp(min=0.0)
            delta = ((-dc - disc.sqrt()) / cc).clamp(0.0, 1.0)
            delta = torch.where(fok, delta, torch.full_like(delta, 0.5))
            self.link.append((q, x, far, fok, d + delta[:, None] * ck, ck, (1 - 2 * delta) / (1 + 2 * delta), 4 / (1 + 2 * delta)))

    def stream(self, g):
        """Pull with walls and the CLI rule; also the momentum-exchange force and torque of the links."""
        h = []
        for q in range(19):
            cx, cy, cz = C[q]
            t = torch.roll(g[q], (cz, cy, cx), (0, 1, 2)) if q else g[0]
            cut = [a for a in range(3) if C[q][a] and not self.per[a]]
            if cut:
                t = t.clone()
                edge = {a: tuple((0 if C[q][a] > 0 else self.n[a] - 1) if 2 - a == k else slice(None) for k in range(3)) for a in cut}
                for a in cut:
                    t[edge[a]] = g[OPP[q]][edge[a]]
                for a in cut:
                    if a == 2 and C[q][2] < 0 and self.wall_u:      # the moving upper wall of z
                        t[edge[a]] += 6.0 * W[q] * C[q][0] * self.wall_u
            h.append(t)
        F = torch.zeros(3, dtype=torch.float64, device=self.dev)
        T = torch.zeros(3, dtype=torch.float64, device=self.dev)
        u = torch.tensor(self.u, device=self.dev)
        w = torch.tensor(self.w, device=self.dev)
        for q, x, far, fok, arm, ck, k0, alpha in self.link:
            k = OPP[q]
            gk, gq = g[k].reshape(-1), g[q].reshape(-1)
            vb = u + torch.linalg.cross(w.expand_as(arm), arm)
            out = gk[x]
            new = out + k0 * torch.where(fok, gk[far], torch.zeros_like(out)) - k0 * gq[x] - alpha * 3.0 * W[k] * (vb @ ck)
            fl = (ck - vb) * (W[k] + out)[:, None] + (ck + vb) * (W[q] + new)[:, None]
            F = F + fl.sum(0)
            T = T + torch.linalg.cross(arm, fl).sum(0)
            h[q] = h[q].reshape(-1).index_put((x,), new).view_as(h[q])
        return h, F, T

    def collide(self, h):
        """TRT of Sec. 2.1, with the two bulk-rate modes of the MRT where the bulk factor is not 1, and a Guo source."""
        tau = self.tau
        sp, sm = 1.0 / tau, 1.0 / (0.5 + MAGIC / (tau - 0.5))
        fluid = (~self.flags).to(torch.float64)
        rho = h[0]
        for q in range(1, 19):
            rho = rho + h[q]
        u = []
        for a in range(3):
            t = 0.0
            for q in range(1, 19):
                if C[q][a]:
                    t = t + h[q] if C[q][a] > 0 else t - h[q]
            u.append(t if self.force is None else t + 0.5 * self.force[a])
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = None if self.force is None else u[0] * self.force[0] + u[1] * self.force[1] + u[2] * self.force[2]
        mrt = self.bulk != 1.0
        out = [None] * 19
        e = W[0] * (rho - 1.5 * uu)
        sums = [h[0] - e, 0.0, 0.0]
        out[0] = h[0] - sp * (h[0] - e)
        if uF is not None:
            out[0] = out[0] + (1 - 0.5 * sp) * W[0] * (-3.0 * uF)
        for q in range(1, 19, 2):
            cu = _dot(C[q], u)
            ep = W[q] * (rho + 4.5 * cu * cu - 1.5 * uu)
            em = 3.0 * W[q] * cu
            hp, hm = 0.5 * (h[q] + h[q + 1]), 0.5 * (h[q] - h[q + 1])
            p, m = hp - sp * (hp - ep), hm - sm * (hm - em)
            if uF is not None:
                cF = _dot(C[q], self.force)
                p = p + (1 - 0.5 * sp) * W[q] * (9.0 * cu * cF - 3.0 * uF)
                m = m + (1 - 0.5 * sm) * W[q] * 3.0 * cF
            out[q], out[q + 1] = p + m, p - m
            if mrt:
                sums[1 if q < 7 else 2] = sums[1 if q < 7 else 2] + 2.0 * (hp - ep)
        if mrt:      # modes |c|^2 - 1 (norm 2/3) and 3|c|^4 - 6|c|^2 + 1 (norm 2), relaxed with s_b instead of s+
            db = 1.0 / (0.5 + self.bulk * (tau - 0.5)) - sp
            c4, c16 = 1.5 * (sums[2] - sums[0]), 0.5 * (sums[0] - 2.0 * sums[1] + sums[2])
            for q in range(19):
                out[q] = out[q] - db * W[q] * ((c16 - c4) if q == 0 else (-2.0 * c16 if q < 7 else c4 + c16))
        return [v * fluid for v in out]

    def advance(self, F, T):
        """Algorithm 1 with the virtual mass of Sec. 3.3 (kick, drift, kick)."""
        Fb = F if self.F_old is None else 0.5 * (F + self.F_old)
        Tb = T if self.T_old is None else 0.5 * (T + self.T_old)
        first = self.F_old is None
        self.F_old, self.T_old = F, T
        m, I = (self.pi + self.cv) * self.V, 0.4 * (self.pi + self.cv) * self.V * self.r ** 2
        self.Fp = Fb + (self.pi - 1.0) * self.gz * self.V + self.cv * self.V * self.a
        Tp = Tb + 0.4 * self.cv * self.V * self.r ** 2 * self.b
        if not self.held:
            self.u = self.u + (0.0 if first else 0.5) * self.Fp / m + 0.5 * self.Fp / m
            self.a = self.Fp / m
            self.x = self.x + self.u
            for a in range(3):
                if self.per[a]:
                    self.x[a] = self.x[a] % self.n[a]
        else:
            self.a = np.zeros(3)
        self.w = self.w + (0.0 if first else 0.5) * Tp / I + 0.5 * Tp / I
        self.b = Tp / I
        self.history.append(np.concatenate((F, T, self.x, self.u, self.w)))

    def remap(self, g):
        """New flags; covered cells dropped, uncovered cells refilled (Sec. 2.3)."""
        if self.held:
            return g
        new = self.solid()
        gone, fresh = new & ~self.flags, ~new & self.flags
        if bool((gone | fresh).any()):
            g = g.reshape(19, -1)
            both = ~(new | self.flags).reshape(-1)
            g[:, gone.reshape(-1)] = 0.0
            cells = self.box_cells(fresh)
            near = [self.at(cells, C[q]) for q in range(1, 19)]
            index = torch.stack([y for y, _ in near], dim=1)
            ok = (torch.stack([k for _, k in near], dim=1) & both[index]).cpu().numpy()
            around = g[:, index.reshape(-1)].view(19, -1, 18).cpu().numpy()
            off = self.offsets()
            pos = torch.stack([off[a][cells[:, a]] for a in range(3)], dim=1).cpu().numpy()
            cv = np.array(C, dtype=np.float64)
            vals = []
            for i in range(len(pos)):
                rs = [1.0 + around[:, i, k].sum() for k in range(18) if ok[i, k]]
                nb = {k + 1: around[:, i, k] @ cv for k in range(6) if ok[i, k]}
                drho = (np.mean(rs) if rs else 1.0) - 1.0
                u = self.u + np.cross(self.w, pos[i])
                e = np.array([W[q] * (drho + 3 * (cv[q] @ u) + 4.5 * (cv[q] @ u) ** 2 - 1.5 * (u @ u)) for q in range(19)])
                if self.grad_refill:
                    G = np.zeros((3, 3))
                    for a in range(3):
                        p, m = nb.get(1 + 2 * a), nb.get(2 + 2 * a)
                        if p is not None and m is not None:
                            G[a] = 0.5 * (p - m)
                        elif p is not None:
                            G[a] = p - u
                        elif m is not None:
                            G[a] = u - m
                    S = 0.5 * (G + G.T)
                    sp = 1.0 / self.tau
                    for q in range(19):
                        e[q] += -3.0 * W[q] * (1.0 - sp) / sp * ((np.outer(cv[q], cv[q]) - np.eye(3) / 3.0) * S).sum()
                vals.append(e)
            if vals:
                x = cells[:, 0] + self.n[0] * (cells[:, 1] + self.n[1] * cells[:, 2])
                g[:, x] = torch.tensor(np.stack(vals, axis=1), device=self.dev)
            g = g.view(19, *reversed(self.n))
            self.flags = new
        self.links()
        return g

    def equilibrium(self, u):
        """The start: density 1 and the velocity field u (None: at rest), nothing inside the sphere."""
        if u is None:
            return torch.zeros((19,) + tuple(reversed(self.n)), dtype=torch.float64, device=self.dev)
        fluid = (~self.flags).to(torch.float64)
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        out = []
        for q in range(19):
            cu = _dot(C[q], u)
            out.append(W[q] * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu) * fluid)
        return torch.stack(out)

    def run(self, g, steps):
        for _ in range(steps):
            h, F, T = self.stream(g)
            del g
            g = torch.stack(self.collide(h))
            del h
            self.advance(F.cpu().numpy(), T.cpu().numpy())
            g = self.remap(g)
        return g

    def record(self):
        last = self.history[-1]
        return np.concatenate((last, self.a, self.b, self.Fp))


def _exact_run(shape, tau, pos, d, pi, cv, g, steps, u, walls=0, wall_u=0.0, bulk=1.0, grad_refill=False, held=False):
    m = _Method(shape, tau, walls, wall_u, bulk, grad_refill)
    m.sphere(pos, d, pi, cv, (0.0, 0.0, -g), held)
    return m, m.run(m.equilibrium(u), steps)


def exact(case, seed):
    c = case
    scale = 2.0 ** FP16_SCALE if c["precision"] == "fp16" else 1.0
    if c["kind"] == "refined":      # the plain dense form steps every cell of the finest lattice: minutes
        return None
    if c["kind"] == "drag":
        return _exact_drag(c, seed)
    if c["kind"] == "batch":
        fields, records = [], []
        for s in _sweep(c, seed):
            m, f = _exact_run((s["edge"],) * 3, s["tau"], s["pos"], s["diameter"], s["density_ratio"], s["cv"],
                              -s["gravity"][2], c["steps"], None)
            fields.append(f.reshape(-1))
            records.append(m.record())
        return {"field": torch.cat(fields) * scale, "particles": np.stack(records)}
    tau, g = _tau_gravity(c)
    shape = (c["nx"], c["ny"], c["nz"])
    m, f = _exact_run(shape, tau, _start(c, seed), c["diameter"], c["density_ratio"], c["cv"], g, c["steps"],
                      _flow(shape, c["amplitude"], seed, c["walls"], c["wall_u"]), c["walls"], c["wall_u"], c["bulk"],
                      c["refill"] == "grad", bool(c["held"]))
    if scale != 1.0:
        f *= scale
    if c["read"] == "particle":
        return {"field": f, "particle": m.record()}
    return {"field": f, "history": np.stack(m.history)}


def _exact_drag(c, seed):
    """J and its gradients by autograd through the plain steps, a checkpoint at each."""
    shape = (c["nx"], c["ny"], c["nz"])
    low = DTYPE[c["precision"]]
    u0 = _flow(shape, workloads.ADJOINT_64["amplitude"], seed, 0, 0.0).to(low).double().requires_grad_()
    tau = torch.tensor(c["tau"], dtype=low).double().cuda().requires_grad_()
    f0 = [0.0, 0.0, 0.0]
    f0[c["axis"]] = c["force"]
    force = torch.tensor(f0, dtype=low).double().cuda().requires_grad_()
    m = _Method(shape, tau, force=force)
    m.sphere(_start(c, seed), c["diameter"], 1.0, 0.0, (0.0, 0.0, 0.0), True)

    def one(g, tau, force):
        m.tau, m.force = tau, force
        h, F, _ = m.stream(g)
        return torch.stack(m.collide(h)), F

    g = m.equilibrium(u0)
    total = 0.0
    for _ in range(c["steps"]):
        g, F = checkpoint(one, g, tau, force, use_reentrant=False)
        total = total + F[c["axis"]]
    J = total / c["steps"]
    gt, gf, gu = torch.autograd.grad(J, (tau, force, u0))
    return {"J": J.detach(), "grad_tau": gt, "grad_force": gf, "grad_u0": gu}
