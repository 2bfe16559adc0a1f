"""The work that is timed: whole passes through the public entry points.

A user of this framework loads particles into a ``Simulation`` and steps it,
reading back fields, particles or energies, or runs the differentiable laser
slab forward and backward.  Every case does one of these from a fixed start:

  plasma    periodic thermal plasmas and counter-streaming beams
  target    a laser pulse on an electron-proton target between absorbing walls
  history   a plasma stepped one step at a time with the energies read back
  gradient  the differentiable laser slab, objective and gradients

A pass restores the start (a device checkpoint, as the differentiable run
restores its segments), takes ``steps`` steps and reads the whole state back
into device memory: nine field arrays and the particles in id order.  FP32
runs hand their values on as FP32 (the C ABI writes FP64).

``exact`` restates the PIC cycle in FP64 torch operations on full arrays,
without the framework's code, and differentiates it by autograd.
"""
import math

import torch

from paper_1503_02464_gb300 import capi, diff
from paper_1503_02464_gb300.sim import Simulation

TAU = 2.0 * math.pi
FIELD_IDS = range(9)  # Ex Ey Ez Bx By Bz Jx Jy Jz


# ---------------------------------------------------------------- the cases
def _plasma(name, dims, n, order, precision, ppc, u_th, steps, drift=0.0, passes=0, gather="momentum", d=0.05,
            dt=0.0):
    n = tuple(n) + (1,) * (3 - len(n))
    return {"name": name, "kind": "plasma", "dims": dims, "nx": n[0], "ny": n[1], "nz": n[2], "order": order,
            "precision": precision, "ppc": ppc, "u_th": u_th, "drift": drift, "steps": steps, "passes": passes,
            "gather": gather, "d": d, "dt": dt or 0.95 * _courant(d, dims)}


def _target(name, dims, n, precision, ppc, x0, x1, density, a0, steps, d, angle=0.0):
    n = tuple(n) + (1,) * (3 - len(n))
    return {"name": name, "kind": "target", "dims": dims, "nx": n[0], "ny": n[1], "nz": n[2], "order": 2,
            "precision": precision, "ppc": ppc, "x0": x0, "x1": x1, "density": density, "a0": a0, "steps": steps,
            "passes": 0, "gather": "momentum", "d": d * TAU, "dt": 0.9 * _courant(d * TAU, dims), "angle": angle}


def _gradient(name, nx, ny, ppc, steps, segment, precision, store_all):
    return {"name": name, "kind": "gradient", "nx": nx, "ny": ny, "ppc": ppc, "steps": steps, "segment": segment,
            "precision": precision, "store_all": store_all}


def _courant(d, dims):
    return d / math.sqrt(dims)


def listed():
    return [
        # the smallest run in use: the 2D periodic plasma of the FP64 parity
        # preset, where launches and latency count
        _plasma("thermal2d_64_fp64", 2, (64, 64), 1, "fp64", 16, 0.01, 100, dt=0.035),
        # an odd 3D grid (no row a multiple of the vector width, ragged tiles)
        # with the linear shape and the optional steps: current smoothing and
        # the energy-conserving gather
        _plasma("smoothed3d_odd", 3, (75, 50, 43), 1, "fp32", 11, 0.05, 20, passes=2, gather="energy"),
        # a hot 2D plasma on an odd grid: particles change cells often
        _plasma("hot2d_odd", 2, (333, 217), 2, "fp32", 25, 0.6, 20),
        # the headline workload: 256^3 cells, 8 electrons per cell, TSC
        _plasma("thermal3d_256", 3, (256, 256, 256), 2, "fp32", 8, 0.05, 20, dt=0.028),
        # the FP64 path on a 3D plasma
        _plasma("thermal3d_fp64", 3, (64, 64, 64), 2, "fp64", 8, 0.05, 20, dt=0.028),
        # counter-streaming beams, 27 per cell each: the scaling problem's
        # plasma on a smaller grid
        _plasma("twostream3d", 3, (128, 128, 64), 2, "fp32", 27, 0.002, 20, drift=0.2, dt=0.028),
        # energies after every step, the read-back of a running simulation
        dict(_plasma("energies3d_128", 3, (128, 128, 128), 2, "fp32", 8, 0.05, 10, dt=0.028), kind="history"),
        # laser-target runs with the pulse at the target: the 2D slab (64 ppc
        # on 40 columns of a 2048 x 1024 grid), the 3D foil at full size and a
        # smaller 2D target hit at 30 degrees
        _target("laser_slab2d", 2, (2048, 1024), "fp32", 64, 1024, 1064, 40.0, 3.0, 20, 0.02),
        _target("laser_foil3d", 3, (512, 256, 256), "fp32", 27, 256, 276, 50.0, 10.0, 20, 0.03),
        _target("oblique_foil2d", 2, (1024, 512), "fp32", 16, 512, 552, 40.0, 3.0, 20, 0.02, angle=math.radians(30)),
        # gradients with respect to the laser amplitude and the density
        # profile: the default differentiable slab with recomputation, and a
        # small FP64 one with every step recorded
        _gradient("slab_gradient", 256, 256, 16, 200, 20, "fp32", False),
        _gradient("slab_gradient_fp64", 120, 64, 8, 60, 20, "fp64", True),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["plasma3", "plasma3", "plasma2", "beams", "history", "target2", "target3", "gradient"])
    precision = "fp64" if rng.random() < 0.25 else "fp32"
    order = 1 if rng.random() < 0.3 else 2
    opts = {}
    if rng.random() < 0.2:
        opts = {"passes": rng.randint(1, 3), "gather": rng.choice(["momentum", "energy"])}
    if kind in ("plasma3", "history", "beams"):
        most = 64 if precision == "fp64" else 160
        n = [logint(16, most) for _ in range(3)]
        if rng.random() < 0.5:
            n[0] = max(16, n[0] // 8 * 8)
        if kind == "beams":
            n = [min(v, 64) for v in n]
            ppc = rng.randint(8, 32) if precision == "fp32" else rng.randint(2, 8)
            return _plasma("", 3, n, 2, precision, ppc, 0.002, 20, drift=rng.choice([0.1, 0.2, 0.3]))
        ppc = rng.randint(1, 16)
        c = _plasma("", 3, n, order, precision, ppc, math.exp(rng.uniform(math.log(0.01), math.log(0.5))),
                    rng.randint(5, 20), **opts)
        return dict(c, kind="history", passes=0) if kind == "history" else c
    if kind == "plasma2":
        most = 256 if precision == "fp64" else 1024
        n = [logint(16, most), logint(16, most)]
        return _plasma("", 2, n, order, precision, rng.randint(1, 64), math.exp(rng.uniform(math.log(0.01), 0.0)),
                       rng.randint(10, 40), **opts)
    if kind == "target2":
        nx, ny = logint(128, 2048), logint(64, 1024)
        x0 = nx // 2
        return _target("", 2, (nx, ny), precision, rng.randint(4, 64), x0, x0 + rng.randint(8, 40), 40.0,
                       rng.uniform(0.5, 8.0), 20, 0.02, angle=rng.choice([0.0, 0.0, math.radians(30)]))
    if kind == "target3":
        nx, ny, nz = logint(64, 256), logint(24, 128), logint(24, 128)
        x0 = nx // 2
        return _target("", 3, (nx, ny, nz), "fp32", rng.randint(4, 27), x0, x0 + rng.randint(4, 20), 50.0,
                       rng.uniform(0.5, 10.0), 20, 0.03)
    segment = rng.choice([10, 20])
    big = precision == "fp32"
    return _gradient("", rng.randint(96, 256 if big else 144), logint(32, 256 if big else 96),
                     rng.randint(2, 16 if big else 8), segment * rng.randint(2, 6), segment, precision,
                     rng.random() < 0.4)


# ------------------------------------------------------------------- inputs
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _cells_uniform(c, x0, x1, ppc, g):
    """Global positions of ppc particles drawn uniformly in every cell of columns [x0, x1)."""
    dims, nx, ny, nz = c["dims"], c["nx"], c["ny"], c["nz"]
    w = x1 - x0
    cells = torch.arange(w * ny * nz, device="cuda", dtype=torch.int64).repeat_interleave(ppc)
    idx = [x0 + cells % w, torch.div(cells, w, rounding_mode="floor") % ny,
           torch.div(cells, w * ny, rounding_mode="floor")]
    del cells
    pos = []
    for a in range(3):
        if a < dims:
            r = torch.rand(idx[a].shape, generator=g, device="cuda", dtype=torch.float64)
            pos.append((idx[a].double() + r) * c["d"])
        else:
            pos.append(torch.zeros(idx[a].shape, device="cuda", dtype=torch.float64))
    return pos


def _momenta(n, u_th, mean, g):
    return [u_th * torch.randn(n, generator=g, device="cuda", dtype=torch.float64) + m for m in mean]


def _species(c, seed):
    """(charge, mass, x, u, w) of every species: position and momentum components and weight as FP64 arrays."""
    dims, ppc = c["dims"], c["ppc"]
    if c["kind"] != "target":
        # electrons over an immobile background, or two beams of half the density
        for i, u0 in enumerate([c["drift"], -c["drift"]] if c["drift"] else [0.0]):
            g = _gen(seed, i)
            x = _cells_uniform(c, 0, c["nx"], ppc, g)
            u = _momenta(x[0].numel(), c["u_th"], (u0, 0.0, 0.0), g)
            dens = 0.5 if c["drift"] else 1.0
            yield -1.0, 1.0, x, u, torch.full_like(x[0], dens / ppc)
        return
    # a neutral target: protons start where the electrons do; the electrons
    # are warm, and hot (1 MeV-like tails) in the first eight columns
    g = _gen(seed)
    x = _cells_uniform(c, c["x0"], c["x1"], ppc, g)
    w = torch.full_like(x[0], c["density"] / ppc)
    u = _momenta(x[0].numel(), 1.0, (0.0, 0.0, 0.0), g)
    th = torch.where(x[0] < (c["x0"] + 8) * c["d"], 0.3, 0.02)
    yield -1.0, 1.0, x, [v * th for v in u], w
    del u, th
    yield 1.0, 1836.0, x, _momenta(x[0].numel(), 1e-4, (0.0, 0.0, 0.0), g), w


def _laser(c):
    """The pulse that enters at x = 0 while an earlier one is at the target."""
    width = c["ny"] * c["d"]
    return {"a0": c["a0"], "waist": 0.25 * width, "duration": 8 * TAU, "pol": 1, "y_center": 0.5 * width,
            "z_center": 0.5 * c["nz"] * c["d"], "angle": c["angle"]}


def _start_fields(c, seed):
    """E and B at the start, (which, array) pairs: thermal noise in a plasma,
    the pulse in front of a target (travelling along +x, damped inside)."""
    shape = (c["nz"], c["ny"], c["nx"])
    if c["kind"] != "target":
        g = _gen(seed, 7)
        for which in range(6):
            yield which, 0.002 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
        return
    g = _gen(seed, 8)
    phase = TAU * float(torch.rand(1, generator=g, device="cuda"))
    ax = [torch.arange(n, device="cuda", dtype=torch.float64) for n in (c["nx"], c["ny"], c["nz"])]
    d, waist, front = c["d"], 0.25 * c["ny"] * c["d"], c["x0"] * c["d"]

    def pulse(ox, oy, oz):
        x, y, z = (ax[0] + ox) * d, (ax[1] + oy - 0.5 * c["ny"]) * d, (ax[2] + oz - 0.5 * c["nz"]) * d
        s = (front - x).clamp(min=0.0)
        length = min(4 * TAU, 0.8 * front)
        env = torch.where(s < length, torch.sin(0.5 * math.pi * (1 - s / length)) ** 2, torch.zeros_like(s))
        env = env * torch.where(x > front, torch.exp(-(x - front) / (3 * d)), torch.ones_like(x))
        r2 = y[:, None] ** 2 if c["dims"] == 2 else z[:, None, None] ** 2 + y[None, :, None] ** 2
        prof = torch.exp(-r2 / waist ** 2)
        return (c["a0"] * prof * (env * torch.sin(x + phase))).reshape(shape)

    yield capi.PIC_EY, pulse(0.0, 0.5, 0.0)
    yield capi.PIC_BZ, pulse(0.5, 0.5, 0.0)


def _slab(case, seed):
    r = _gen(seed, 9)
    amp = torch.rand(2, generator=r, device="cuda", dtype=torch.float64).tolist()
    # the slab stands where the pulse arrives after about half of the steps;
    # long runs look at the electrons behind it, short ones at its own too
    k = max(8, int(0.32 * case["steps"]))
    first = k + 20 if case["steps"] >= 160 else k
    run = diff.SlabRun(nx=case["nx"], ny=case["ny"], ppc=case["ppc"], steps=case["steps"], segment=case["segment"],
                       slab=(k, k + 20), obj=(first, k + 52), seed=1005 + int(seed) % 100000,
                       waist=0.25 * case["ny"] * 0.05 * TAU, precision=case["precision"],
                       store_all=case["store_all"])
    prof = run.default_profile()
    prof[k:k + 20] *= torch.linspace(0.6, 1.0, 20, dtype=torch.float64).numpy() * (0.8 + 0.4 * amp[0])
    return run, 1.5 + amp[1], prof


def _out_dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


# ------------------------------------------------------------ prepare / run
def prepare(case, seed):
    if case["kind"] == "gradient":
        run_, a0, prof = _slab(case, seed)
        sim = diff.build_sim(run_, a0, prof)
        sim.checkpoint(run_.steps)  # a slot that the run itself does not use
        return {"case": case, "slab": run_, "sim": sim}
    c = case
    n = (c["nx"], c["ny"], c["nz"])
    sim = Simulation(c["dims"], n, (c["d"],) * 3, c["dt"], c["order"], c["precision"],
                     absorbing_x=c["kind"] == "target", laser=_laser(c) if c["kind"] == "target" else None,
                     filter_passes=c["passes"], filter_compensate=c["passes"] > 1, gather=c["gather"])
    counts = []
    for q, m, x, u, w in _species(c, seed):
        k = sim.add_species(q, m, x[0].numel())
        sim.load(k, {"x": x[0], "y": x[1], "z": x[2], "ux": u[0], "uy": u[1], "uz": u[2], "w": w})
        sim._keep = None  # the library has copied the arrays
        counts.append(x[0].numel())
    for which, f in _start_fields(c, seed):
        capi.pic_set_field(sim.h, which, f.data_ptr(), capi.PIC_MEM_DEVICE)
    state = {"case": case, "sim": sim}
    sim.checkpoint(0)
    if c["kind"] != "history":
        # read-back buffers that the program keeps: a species' slots hold up
        # to three padding slots per tile
        t = (16, 16, 1) if c["dims"] == 2 else (8, 8, 4)
        pad = 3 * math.prod(-(-n[a] // t[a]) for a in range(3))
        most = max(counts) + pad
        state["f64"] = [torch.empty(most, dtype=torch.float64, device="cuda") for _ in range(6)]
        state["i32"] = [torch.empty(most, dtype=torch.int32, device="cuda") for _ in range(2)]
        state["counts"] = counts
    return state


def run(state):
    c, sim = state["case"], state["sim"]
    if c["kind"] == "gradient":
        slab = state["slab"]
        sim.restore(slab.steps)
        F = diff.run_forward(slab, sim)
        da0, dprof = diff.backward_gradients(slab, sim)
        dt = _out_dtype(c)
        return {"F": torch.tensor(F, dtype=dt), "da0": torch.tensor(da0, dtype=dt),
                "dprofile": torch.from_numpy(dprof).to(dt)}
    sim.restore(0)
    if c["kind"] == "history":
        rows = []
        for _ in range(c["steps"]):
            sim.step(1)
            e = sim.energy()
            rows.append([e["energy_e"], e["energy_b"], e["energy_kinetic"]])
        return {"energies": torch.tensor(rows, dtype=_out_dtype(c)), "alive": e["n_alive"]}
    sim.step(c["steps"])
    out = {"fields": [sim.field_device(k).to(_out_dtype(c)) for k in FIELD_IDS]}
    for k, count in enumerate(state["counts"]):
        out["species%d" % k] = _particles(state, k, count)
    return out


def _particles(state, k, count):
    """Positions and momenta of one species in id order (zero where a particle left through a wall)."""
    c, sim = state["case"], state["sim"]
    n = sim.num_particles(k)
    buf, (ids, alive) = state["f64"], state["i32"]
    ptr = [b.data_ptr() for b in buf]
    capi.pic_particles(sim.h, k, *ptr, None, ids.data_ptr(), alive.data_ptr(), capi.PIC_MEM_DEVICE)
    live = alive[:n] > 0
    at = torch.where(live, ids[:n].long(), count)  # dead slots: one place past the end
    res = []
    for a in range(6):
        if a == 2 and c["dims"] == 2:
            continue
        o = torch.zeros(count + 1, dtype=_out_dtype(c), device="cuda")
        o.index_copy_(0, at, buf[a][:n].to(o.dtype))
        res.append(o[:count])
    return res


# --------------------------------------------------------------------- work
def _parts(case):
    if case["kind"] == "gradient":
        return (case["nx"] - 7) * case["ny"] * case["ppc"]
    if case["kind"] == "target":
        return 2 * (case["x1"] - case["x0"]) * case["ny"] * case["nz"] * case["ppc"]
    return case["nx"] * case["ny"] * case["nz"] * case["ppc"] * (2 if case["drift"] else 1)


def work(case):
    """Per step every particle's cell, offsets and momenta are read and
    written and its weight read, and every cell's E and B are read and
    written; the state is read back once.  Flops per particle-step as counted
    by hand for the compact stencils (gather, Boris, move, deposit)."""
    r = 8 if case["precision"] == "fp64" else 4
    flops = {(3, 2): 1117, (3, 1): 496, (2, 2): 445, (2, 1): 251}
    parts, steps = _parts(case), case["steps"]
    if case["kind"] == "gradient":
        cells = case["nx"] * case["ny"]
        # forward once, and a reverse step reads the recorded state and
        # updates the adjoints of position, momentum and weight
        step_b = parts * (2 * (4 + 5 * r) + r) + cells * 12 * r
        back_b = parts * (8 + 6 * r + 2 * (5 * r + 8)) + cells * (6 * r + 2 * 6 * r)
        return {"bytes": steps * (step_b + back_b), "flops": steps * parts * 3.5 * flops[2, 2]}
    dims, cells = case["dims"], case["nx"] * case["ny"] * case["nz"]
    step_b = parts * (2 * (4 + (dims + 3) * r) + r) + cells * 12 * r
    out_b = 16 * steps if case["kind"] == "history" else parts * (dims + 3) * r + cells * 9 * r
    return {"bytes": steps * step_b + out_b, "flops": steps * parts * flops[dims, case["order"]]}


# -------------------------------------------------------------------- exact
# The PIC cycle on full arrays in FP64.  A species is a dict of per-axis
# integer cells i, offsets f in [0, 1), momenta u, weight w and a live mask;
# fields are flat arrays, x fastest.
class _Cycle:
    def __init__(self, dims, n, d, dt, order, passes=0, compensate=False, gather="momentum", walls=False,
                 laser=None):
        self.dims, self.n, self.d, self.dt, self.order = dims, n, d, dt, order
        self.passes, self.compensate, self.lower = passes, compensate, gather == "energy"
        self.walls, self.laser = walls, laser

    @staticmethod
    def spline(order, x):
        a = x.abs()
        if order == 0:
            return ((x >= -0.5) & (x < 0.5)).to(x.dtype)
        if order == 1:
            return (1.0 - a).clamp(min=0.0)
        return torch.where(a < 0.5, 0.75 - x * x, 0.5 * (1.5 - a).clamp(min=0.0) ** 2)

    def stencil(self, f, half):
        """(first node, weights) of one axis at offset f, for nodes at integer or half-integer positions."""
        order = self.order - (1 if half and self.lower else 0)
        x = f - 0.5 if half else f
        first = torch.floor(x if order == 1 else x + 0.5) - (1 if order == 2 else 0)
        if order == 0:  # nearest half-integer node of the particle's own cell
            first = torch.zeros_like(first)
            return first.long(), [torch.ones_like(x)]
        return first.long(), [self.spline(order, x - (first + k)) for k in range(order + 1)]

    def index(self, i, first, k, axis):
        return (i[axis] + first + k) % self.n[axis]

    def gathered(self, sp, F, half):
        idx, wts = [], []
        for a in range(self.dims):
            first, w = self.stencil(sp["f"][a], half[a])
            idx.append([self.index(sp["i"], first, k, a) for k in range(len(w))])
            wts.append(w)
        acc = 0.0
        zs = range(len(wts[2])) if self.dims == 3 else [None]
        for kz in zs:
            for ky in range(len(wts[1])):
                row = idx[1][ky] if kz is None else idx[2][kz] * self.n[1] + idx[1][ky]
                r = sum(F[row * self.n[0] + idx[0][kx]] * wts[0][kx] for kx in range(len(wts[0])))
                acc = acc + r * (wts[1][ky] if kz is None else wts[1][ky] * wts[2][kz])
        return acc

    def push(self, sp, q, m, E, B, J):
        """Moves one species and returns it with J added to."""
        t, h_ = True, False
        e = [self.gathered(sp, E[k], s) for k, s in enumerate([(t, h_, h_), (h_, t, h_), (h_, h_, t)])]
        b = [self.gathered(sp, B[k], s) for k, s in enumerate([(h_, t, t), (t, h_, t), (t, t, h_)])]
        h = q * self.dt / (2.0 * m)
        um = [sp["u"][a] + h * e[a] for a in range(3)]
        gm = torch.sqrt(1.0 + um[0] ** 2 + um[1] ** 2 + um[2] ** 2)
        tv = [h * b[a] / gm for a in range(3)]
        s = 2.0 / (1.0 + tv[0] ** 2 + tv[1] ** 2 + tv[2] ** 2)

        def cross(p, r):
            return [p[1] * r[2] - p[2] * r[1], p[2] * r[0] - p[0] * r[2], p[0] * r[1] - p[1] * r[0]]
        up = [x + y for x, y in zip(um, cross(um, tv))]
        u = [x + s * y + h * z for x, y, z in zip(um, cross(up, tv), e)]
        gam = torch.sqrt(1.0 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        x1 = [sp["f"][a] + self.dt / self.d[a] * u[a] / gam for a in range(self.dims)]
        J = self.deposit(sp, x1, u[2] / gam, q, J)
        fl = [torch.floor(v.detach()) for v in x1]
        i = [(sp["i"][a] + fl[a].long()) % self.n[a] if a < self.dims else sp["i"][a] for a in range(3)]
        f = [x1[a] - fl[a] for a in range(self.dims)]
        live = sp["live"]
        if self.walls:
            X = sp["i"][0] + x1[0].detach()
            live = live & (X >= 3.0) & (X < self.n[0] - 4.0)
        return {"i": i, "f": f, "u": u, "w": sp["w"], "live": live}, J

    def deposit(self, sp, x1, vz, q, J):
        nw = self.order + 2
        S0, DS, idx = [], [], []
        for a in range(self.dims):
            f = sp["f"][a]
            lo = torch.minimum(f.detach(), x1[a].detach())
            first = torch.floor(lo + 0.5) - 1 if self.order == 2 else torch.floor(lo)
            s0 = [self.spline(self.order, f - (first + k)) for k in range(nw)]
            s1 = [self.spline(self.order, x1[a] - (first + k)) for k in range(nw)]
            S0.append(s0)
            DS.append([p - r for p, r in zip(s1, s0)])
            idx.append([self.index(sp["i"], first.long(), k, a) for k in range(nw)])
        w = torch.where(sp["live"], sp["w"], torch.zeros_like(sp["w"]))
        J = list(J)
        run = []
        for a in range(self.dims):
            c, acc = [], 0.0
            for k in range(nw - 1):
                acc = acc + DS[a][k]
                c.append(-q * self.d[a] / self.dt * w * acc)
            run.append(c)
        n0, n1 = self.n[0], self.n[1]
        if self.dims == 2:
            for b in range(nw):
                for a in range(nw):
                    at = idx[1][b] * n0 + idx[0][a]
                    if a < nw - 1:
                        J[0] = J[0].index_add(0, at, run[0][a] * (S0[1][b] + 0.5 * DS[1][b]))
                    if b < nw - 1:
                        J[1] = J[1].index_add(0, at, run[1][b] * (S0[0][a] + 0.5 * DS[0][a]))
                    J[2] = J[2].index_add(0, at, q * w * vz * (
                        S0[0][a] * (S0[1][b] + 0.5 * DS[1][b]) + DS[0][a] * (0.5 * S0[1][b] + DS[1][b] / 3.0)))
            return J

        def mean(p, r, k, l):
            return S0[p][k] * (S0[r][l] + 0.5 * DS[r][l]) + DS[p][k] * (0.5 * S0[r][l] + DS[r][l] / 3.0)
        for c in range(nw):
            for b in range(nw):
                for a in range(nw):
                    at = (idx[2][c] * n1 + idx[1][b]) * n0 + idx[0][a]
                    if a < nw - 1:
                        J[0] = J[0].index_add(0, at, run[0][a] * mean(1, 2, b, c))
                    if b < nw - 1:
                        J[1] = J[1].index_add(0, at, run[1][b] * mean(2, 0, c, a))
                    if c < nw - 1:
                        J[2] = J[2].index_add(0, at, run[2][c] * mean(0, 1, a, b))
        return J

    def smooth(self, j):
        v = j.view(self.n[2], self.n[1], self.n[0])
        alphas = [0.5] * self.passes + ([1.0 + 0.5 * self.passes] if self.compensate else [])
        for al in alphas:
            for ax in (2, 1, 0)[:self.dims]:
                v = al * v + 0.5 * (1 - al) * (torch.roll(v, 1, ax) + torch.roll(v, -1, ax))
        return v.reshape(-1)

    def curl(self, F, way):
        """curl on the Yee lattice; way = -1: forward differences (E at the B places), +1: backward."""
        V = [f.view(self.n[2], self.n[1], self.n[0]) for f in F]

        def dif(v, axis):
            if axis == 2 and self.dims == 2:
                return torch.zeros_like(v)
            return (torch.roll(v, way, 2 - axis) - v) * (-way) / self.d[axis]
        return [(dif(V[2], 1) - dif(V[1], 2)), (dif(V[0], 2) - dif(V[2], 0)), (dif(V[1], 0) - dif(V[0], 1))]

    def half_b(self, E, B):
        c = self.curl(E, -1)
        out = []
        for k in range(3):
            g = c[k]
            if self.walls and k > 0:
                mask = torch.ones(self.n[0], dtype=g.dtype, device=g.device)
                mask[-1] = 0.0
                g = g * mask
            out.append(B[k] - 0.5 * self.dt * g.reshape(-1))
        return out

    def wave(self, t, comp, dev):
        """The incoming wave's (x = 0, x = dx) values at the wall rows of component comp (1 = Ey, 2 = Ez)."""
        L = self.laser
        if not L or L["pol"] != comp:
            return 0.0, 0.0
        y = (torch.arange(self.n[1], device=dev, dtype=torch.float64) + (0.5 if comp == 1 else 0.0)) * self.d[1]
        z = (torch.arange(self.n[2], device=dev, dtype=torch.float64) + (0.5 if comp == 2 else 0.0)) * self.d[2]
        co, si = math.cos(L["angle"]), math.sin(L["angle"])
        y0 = 0.0 if L["angle"] > 0 else self.n[1] * self.d[1] if L["angle"] < 0 else 0.0
        r = []
        for x in (0.0, self.d[0]):
            tau = t - x * co - (y - y0) * si
            rp = (y - L["y_center"]) * co - (x * si if si else 0.0)
            r2 = rp[None, :] ** 2 + ((z[:, None] - L["z_center"]) ** 2 if self.dims == 3 else 0.0)
            env = torch.sin(math.pi * tau / L["duration"]) ** 2 * torch.sin(tau)
            env = torch.where((tau > 0) & (tau < L["duration"]), env, torch.zeros_like(env))
            amp = L["a0"] * (co if comp == 1 and L["angle"] else 1.0)
            r.append(amp * torch.exp(-r2 / L["waist"] ** 2) * env[None, :])
        return r

    def fields(self, E, B, J, t):
        B = self.half_b(E, B)
        c = self.curl(B, 1)
        new = []
        for k in range(3):
            g = self.dt * (c[k] - J[k].view_as(c[k]))
            old = E[k].view_as(c[k])
            if self.walls:
                mask = torch.ones(self.n[0], dtype=g.dtype, device=g.device)
                mask[-1] = 0.0
                if k > 0:
                    mask[0] = 0.0
                g = g * mask
            e = old + g
            if self.walls and k > 0:
                kc = (self.dt - self.d[0]) / (self.dt + self.d[0])
                l0o, l1o = self.wave(t, k, e.device)
                l0n, l1n = self.wave(t + self.dt, k, e.device)
                left = l0n + (old[..., 1] - l1o) + kc * ((e[..., 1] - l1n) - (old[..., 0] - l0o))
                right = old[..., -2] + kc * (e[..., -2] - old[..., -1])
                e = torch.cat([left[..., None], e[..., 1:-1], right[..., None]], -1)
            new.append(e.reshape(-1))
        return new, self.half_b(new, B)

    def step(self, species, charges, E, B, t):
        J = [torch.zeros_like(E[0]) for _ in range(3)]
        moved = []
        for sp, (q, m) in zip(species, charges):
            sp, J = self.push(sp, q, m, E, B, J)
            moved.append(sp)
        if self.passes:
            J = [self.smooth(j) for j in J]
        E, B = self.fields(E, B, J, t)
        return moved, E, B, J


def _placed(cy, x, u, w):
    i, f = [], []
    for a in range(3):
        if a >= cy.dims:
            i.append(torch.zeros(x[0].shape, dtype=torch.int64, device=x[0].device))
            continue
        s = x[a] / cy.d[a]
        fl = torch.floor(s)
        i.append(fl.long() % cy.n[a])
        f.append(s - fl)
    live = torch.ones(x[0].shape, dtype=torch.bool, device=x[0].device)
    if cy.walls:
        s = x[0] / cy.d[0]
        live = (s >= 3.0) & (s < cy.n[0] - 4.0)
    return {"i": i, "f": f, "u": list(u), "w": w, "live": live}


def exact(case, seed):
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed)
    c = case
    nodes = (c["order"] + 2) ** c["dims"]
    if _parts(c) * c["steps"] * nodes > 3e10:
        return None  # beyond about 20 s
    cy = _Cycle(c["dims"], (c["nx"], c["ny"], c["nz"]), (c["d"],) * 2 + (c["d"] if c["dims"] == 3 else 1.0,), c["dt"],
                c["order"], c["passes"], c["passes"] > 1, c["gather"], c["kind"] == "target",
                _laser(c) if c["kind"] == "target" else None)
    species, charges = [], []
    for q, m, x, u, w in _species(c, seed):
        species.append(_placed(cy, x, u, w))
        charges.append((q, m))
    F = [torch.zeros(c["nx"] * c["ny"] * c["nz"], dtype=torch.float64, device="cuda") for _ in range(6)]
    for which, f in _start_fields(c, seed):
        F[which] = f.reshape(-1).clone()
    E, B = F[:3], F[3:]
    dV = math.prod(cy.d)
    rows = []
    with torch.no_grad():
        for t in range(c["steps"]):
            species, E, B, J = cy.step(species, charges, E, B, t * c["dt"])
            if c["kind"] == "history":
                kin = 0.0
                for sp, (q, m) in zip(species, charges):
                    u2 = sp["u"][0] ** 2 + sp["u"][1] ** 2 + sp["u"][2] ** 2
                    kin += float((sp["w"] * u2 / (torch.sqrt(1 + u2) + 1)).sum()) * m * dV
                rows.append([0.5 * dV * sum(float((e * e).sum()) for e in E),
                             0.5 * dV * sum(float((b * b).sum()) for b in B), kin])
    if c["kind"] == "history":
        return {"energies": torch.tensor(rows, dtype=torch.float64), "alive": None}
    shape = (c["nz"], c["ny"], c["nx"])
    out = {"fields": [f.view(shape) for f in E + B + list(J)]}
    for k, sp in enumerate(species):
        keep = sp["live"].double()
        x = [(sp["i"][a] + sp["f"][a]) * cy.d[a] * keep for a in range(c["dims"])]
        out["species%d" % k] = x + [u * keep for u in sp["u"]]
    return out


def _exact_gradient(case, seed):
    from torch.utils.checkpoint import checkpoint
    run_, a0, prof = _slab(case, seed)
    if _parts(case) * case["steps"] > 1.2e8:
        return None  # beyond about 20 s
    d = run_.d
    parts = run_.particles(prof)
    amp = torch.tensor(a0, dtype=torch.float64, device="cuda", requires_grad=True)
    profile = torch.tensor(prof, dtype=torch.float64, device="cuda", requires_grad=True)
    cy = _Cycle(2, (run_.nx, run_.ny, 1), (d, d, 1.0), run_.dt, 2, walls=True,
                laser={"a0": amp, "waist": run_.waist, "duration": run_.duration, "pol": 1, "angle": 0.0,
                       "y_center": 0.5 * run_.ny * d, "z_center": 0.5})
    x, u = ([torch.from_numpy(parts[k]).cuda() for k in ks] for ks in (("x", "y", "z"), ("ux", "uy", "uz")))
    cols = torch.from_numpy(run_.column_of_id(parts["id"]).astype("int64")).cuda()
    sp = _placed(cy, x, u, profile[cols] / run_.ppc)
    F = [torch.zeros(run_.nx * run_.ny, dtype=torch.float64, device="cuda") for _ in range(6)]

    def one(t, E, B, sp):
        (sp,), E, B, _ = cy.step([sp], [(-1.0, 1.0)], E, B, t)
        return E, B, sp
    E, B = F[:3], F[3:]
    for k in range(run_.steps):
        E, B, sp = checkpoint(one, k * run_.dt, E, B, sp, use_reentrant=False)
    u2 = sp["u"][0] ** 2 + sp["u"][1] ** 2 + sp["u"][2] ** 2
    inside = sp["live"] & (sp["i"][0] >= run_.obj[0]) & (sp["i"][0] < run_.obj[1])
    obj = (sp["w"] * u2 / (torch.sqrt(1 + u2) + 1) * inside.double()).sum() * d * d
    obj.backward()
    return {"F": obj.detach(), "da0": amp.grad, "dprofile": profile.grad}
