"""Performance cases of the time step: what a program that uses this package has it do.

A case is a dict of plain values; ``listed()`` names the standing ones, ``draw(rng)`` gives
further ones of the same ranges.  ``prepare`` makes a handle and its inputs, ``run`` is one
pass through the public entry points (``capi.Sim``, the C ABI), ``work`` is the least the
pass has to move and compute, ``exact`` is its answer in 64 bits from plain numpy.

Kinds of pass:
  run      ``steps`` time steps of a plasma, then the diagnostics of every instance (the
           loop of a production run: step, moments, step, moments).  With ``fresh`` the
           pass starts from its initial particles again, loaded from device memory (a short
           run or a parameter scan on one handle).
  restart  a checkpoint of a periodic plasma taken up: particles with their collision clocks
           from host memory, the counters restored, a few steps, and the particles read back
           to host memory (the next checkpoint).
  field    the allocation-free field solve on a charge deposit that is already on the device.

Plasmas (``workloads``): ``bounded`` between absorbing walls, ``source`` magnetized with a
volume source and ionization, ``ionization`` the periodic test case of e, D+ and D particles,
``ensemble`` a batch of uneven ``source`` instances.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2404_10270_gb300 import capi, workloads as W

SORT = 20
DX, DT, T_N = 0.5, 0.05, 0.05
M_ION, NU, E_EXT = 100.0, 0.01, 0.05
RESTART_STEP = 50
DIAGNOSTICS = ("step", "live", "wall_count", "wall_energy", "collisions", "kinetic", "next_id",
               "density", "phi", "E")


def listed():
    return [
        # the smallest plasma of the benchmark, where launches and latency count: a short
        # run from its load, in both precisions (the second ragged, with the smoother)
        dict(name="small_f32", kind="run", plasma="bounded", cells=256, ppc=100, precision="f32",
             steps=100, fresh=True, ion_nstep=1, smooth=0, block=256),
        dict(name="small_f64_smooth", kind="run", plasma="bounded", cells=333, ppc=77,
             precision="f64", steps=97, fresh=True, ion_nstep=1, smooth=1, block=256),
        # the headline workload: 196.6 M particles, one sort cycle between diagnostics
        dict(name="bounded_f32", kind="run", plasma="bounded", cells=65536, ppc=1500,
             precision="f32", steps=20, fresh=False, ion_nstep=1, smooth=0, block=512),
        dict(name="bounded_f64", kind="run", plasma="bounded", cells=65536, ppc=1500,
             precision="f64", steps=20, fresh=False, ion_nstep=1, smooth=0, block=512),
        # heavy ions moved every fourth step, a ragged size
        dict(name="subcycled_f32", kind="run", plasma="bounded", cells=30011, ppc=701,
             precision="f32", steps=20, fresh=False, ion_nstep=4, smooth=0, block=256),
        # the paper's own test case: neutral particle targets that ionization depletes
        dict(name="ionization_f32", kind="run", plasma="ionization", cells=100000, ppc=100,
             precision="f32", steps=20, fresh=False, block=256),
        dict(name="ionization_f64", kind="run", plasma="ionization", cells=100000, ppc=100,
             precision="f64", steps=20, fresh=False, block=256),
        # one magnetized plasma with a volume source, double precision, run from its load
        dict(name="source_f64", kind="run", plasma="source", cells=4096, ppc=200,
             precision="f64", steps=40, fresh=True, ion_nstep=1, block=256),
        # batches of uneven plasmas, every instance's diagnostics read
        dict(name="ensemble_f32", kind="run", plasma="ensemble", instances=128, precision="f32",
             steps=20, fresh=False, block=256),
        dict(name="ensemble_f64", kind="run", plasma="ensemble", instances=40, precision="f64",
             steps=20, fresh=False, block=256),
        # a checkpoint taken up and the next one written, through pageable host memory
        dict(name="restart_f64", kind="restart", cells=25003, ppc=40, precision="f64", steps=4),
        # the field solve of callers that own all device memory, at the largest size it takes
        dict(name="field_65536", kind="field", cells=65536, ppc=1500, precision="f32"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("bounded", "bounded", "bounded", "ionization", "source", "ensemble",
                       "restart", "field"))
    precision = rng.choice(("f32", "f64"))
    if kind == "field":
        return dict(kind="field", cells=log_int(64, 65536), ppc=log_int(20, 1500),
                    precision=precision)
    if kind == "restart":
        cells = log_int(256, 50000)
        return dict(kind="restart", cells=cells, ppc=min(log_int(20, 400), 2000000 // cells),
                    precision=precision, steps=rng.randint(2, 8))
    if kind == "ensemble":
        return dict(kind="run", plasma="ensemble", instances=log_int(24, 128),
                    precision=precision, steps=20, fresh=False, block=256)
    if kind == "ionization":
        cells = log_int(20000, 130000)
        return dict(kind="run", plasma="ionization", cells=cells, ppc=rng.randint(60, 160),
                    precision=precision, steps=20, fresh=False, block=256)
    if kind == "source":
        return dict(kind="run", plasma="source", cells=log_int(256, 8192),
                    ppc=rng.randint(50, 400), precision=precision, steps=rng.randint(20, 60),
                    fresh=True, ion_nstep=1, block=256)
    cells = log_int(64, 65536)
    ppc = min(log_int(20, 1500), 30000000 // cells)
    large = 2 * cells * ppc >= 4000000
    return dict(kind="run", plasma="bounded", cells=cells, ppc=ppc, precision=precision,
                steps=SORT if large else rng.randint(20, 100), fresh=not large,
                ion_nstep=rng.choice((1, 1, 4)), smooth=rng.choice((0, 0, 1)), block=256)


def _physics(case, seed):
    """The instances of a run or restart case; the Philox keys come from the seed."""
    plasma = case.get("plasma", "bounded")
    if plasma == "ensemble":
        # twice the particles may be created before a segment is full
        physs = W.ensemble(case["instances"], key=0, capacity_factor=2.0)
    elif plasma == "ionization":
        physs = [W.ionization_case(case["cells"], case["ppc"], sort_interval=SORT)]
    elif plasma == "source":
        physs = [W.magnetized_source(case["cells"], case["ppc"], ion_nstep=case["ion_nstep"])]
    else:
        physs = [W.bounded_small(case["cells"], case["ppc"], m_i=M_ION, nu=NU, dx=DX, dt=DT,
                                 ion_nstep=case.get("ion_nstep", 1))]
        physs[0].smooth = case.get("smooth", 0)
    if case["kind"] == "restart":
        physs[0].bc, physs[0].field = W.BC_PERIODIC, W.FIELD_EXTERNAL
        physs[0].E_ext = E_EXT
    for i, p in enumerate(physs):
        p.seed = 1 + i + 4096 * (seed % 1000003)
    return physs


def _generator(seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    return torch.Generator(device=device).manual_seed(int(seed)), device


def _particles(species, ncells, precision, gen, device):
    """Exactly ppc particles in each cell, uniform offsets, Maxwellian velocities; species:
    (ppc, thermal speed) pairs.  Ids are species-major."""
    t = torch.float32 if precision == "f32" else torch.float64
    out, next_id = [], 0
    for ppc, vth in species:
        n = ppc * ncells
        cell = torch.arange(ncells, dtype=torch.int32, device=device).repeat_interleave(ppc)
        off = torch.rand(n, generator=gen, device=device, dtype=t)
        v = [torch.randn(n, generator=gen, device=device, dtype=t).mul_(vth) for _ in range(3)]
        ids = torch.arange(next_id, next_id + n, dtype=torch.int32, device=device)
        out.append(W.Load(cell, off, *v, ids))
        next_id += n
    return out


def _species(phys):
    return [(s.ppc, math.sqrt(s.temperature / s.mass)) for s in phys.species]


def _sim(case, physs, block=256):
    return capi.Sim(physs, precision=capi.FP32 if case["precision"] == "f32" else capi.FP64,
                    sort_interval=SORT, block=case.get("block", block))


# ---- a checkpoint ------------------------------------------------------------------------
def _checkpoint(case, seed):
    """Particles of both species in cells per step with their collision clocks at step
    RESTART_STEP, in host memory: a clock either waits for the common test at step 127 or,
    for the share of particles whose candidate comes before it, names that candidate."""
    gen, device = _generator(seed)
    scale = DT / DX
    loads = _particles([(case["ppc"], scale), (case["ppc"], scale / math.sqrt(M_ION))],
                       case["cells"], case["precision"], gen, device)
    wait = 127 - RESTART_STEP
    share = 1.0 - math.exp(-NU * DT * wait)
    for ld in loads:
        n = len(ld.cell)
        pending = torch.rand(n, generator=gen, device=device) < share
        skip = torch.randint(0, wait, (n,), generator=gen, device=device)
        ld.state = torch.where(pending, skip + 128, torch.full_like(skip, wait)).to(torch.uint8)
        for k in ("cell", "off", "vx", "vy", "vz", "id", "state"):
            a = getattr(ld, k).cpu().numpy()
            setattr(ld, k, a.view(np.uint32) if k == "id" else a)
    return loads


# ---- the field solve ---------------------------------------------------------------------
def _deposit(case, seed):
    """Node deposits of two species of ppc particles a cell with their Poisson noise."""
    gen, device = _generator(seed)
    unit = 1 << (24 if case["precision"] == "f32" else 48)
    mean = case["ppc"] * float(unit)
    noise = torch.randn(2, case["cells"] + 1, generator=gen, device=device, dtype=torch.float64)
    charge = (mean + noise * (mean / math.sqrt(case["ppc"]))).clamp_(min=0.0).to(torch.int64)
    charge[:, 0] //= 2
    charge[:, -1] //= 2
    return charge, unit


def prepare(case, seed):
    if case["kind"] == "field":
        charge, unit = _deposit(case, seed)
        return dict(case=case, charge=charge, unit=unit, z=(ctypes.c_int32 * 2)(-1, 1),
                    delta=DX / case["ppc"],
                    E=torch.empty(case["cells"] + 1, dtype=torch.float64, device=charge.device))
    physs = _physics(case, seed)
    if case["kind"] == "restart":
        return dict(case=case, sim=_sim(case, physs), loads=_checkpoint(case, seed))
    sim = _sim(case, physs)
    gen, device = _generator(seed)
    loads = []
    for i, p in enumerate(physs):
        loads.append(_particles(_species(p), p.ncells, case["precision"], gen, device))
    torch.cuda.synchronize()  # the handle's stream is its own
    for i, load in enumerate(loads):
        sim.load_all(load, inst=i)
    return dict(case=case, sim=sim, loads=loads if case["fresh"] else None)


def run(state):
    case = state["case"]
    if case["kind"] == "field":
        charge = state["charge"]
        rc = capi.lib().pic_field_solve_noalloc(
            case["cells"], 2, charge.data_ptr(), state["z"], state["delta"], state["unit"], 1.0,
            state["E"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != 0:
            raise capi.PicError(rc, str(capi.lib().pic_last_error(None)))
        return state["E"]
    sim = state["sim"]
    if case["kind"] == "restart":
        loads = state["loads"]
        for s, ld in enumerate(loads):
            sim.load(0, s, ld, cell_units=True)
        sim.restore_counters(RESTART_STEP, [sum(len(ld) for ld in loads)])
        sim.step(case["steps"])
        dtype = np.float32 if case["precision"] == "f32" else np.float64
        return [sim.particles(0, s, cell_units=True, dtype=dtype) for s in range(len(loads))]
    if case["fresh"]:
        for i, load in enumerate(state["loads"]):
            sim.load_all(load, inst=i)
    sim.step(case["steps"])
    m = [sim.moments(i) for i in range(len(sim.phys))]
    if len(m) == 1:
        return m[0]
    return {k: np.concatenate([np.ravel(x[k]) for x in m]) for k in DIAGNOSTICS}


def work(case):
    """Bytes: in every step each particle's position and the velocities its push changes,
    read and written once (with the cell word), a species that rests in the step none; the
    diagnostics read every particle's cell and velocities; a load, a checkpoint and a
    read-back move every value of a particle once.  Node arrays count once a step."""
    t = 4 if case["precision"] == "f32" else 8
    if case["kind"] == "field":
        return dict(bytes=(2 * 8 + 8) * (case["cells"] + 1.0), flops=10.0 * case["cells"])
    particle = 4 + 4 * t + 4 + 1  # cell, offset, velocities, id, clock
    nbytes = flops = 0.0
    for p in _physics(case, 1):
        mag = any(b != 0.0 for b in p.B)
        for s in p.species:
            n = float(s.ppc * p.ncells)
            moves = case["steps"] / s.nstep
            nbytes += moves * n * 2 * (4 + (4 if mag else 2) * t)
            nbytes += case["steps"] * 3 * 8.0 * (p.ncells + 1)
            flops += moves * n * (40 if mag else 10)
            if case["kind"] == "restart" or case["fresh"]:
                nbytes += 2 * n * particle
            nbytes += n * (2 * particle if case["kind"] == "restart" else 4 + 3 * t)
    return dict(bytes=nbytes, flops=flops)


# ---- the answers in 64 bits --------------------------------------------------------------
def _philox(ids, step, purpose, key):
    """Philox4x32-10 (Salmon et al., SC'11) on counters (id, step_hi, step_lo, purpose)."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [ids.astype(np.uint64), np.full(ids.shape, step >> 32, np.uint64),
         np.full(ids.shape, step & 0xFFFFFFFF, np.uint64),
         np.full(ids.shape, purpose, np.uint64)]
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _uniform(w):
    return (w.astype(np.float64) + 0.5) * 2.0 ** -32


def _solve(rho, n, dx, smooth):
    """phi and E between grounded walls from the node charge densities (half-cell densities
    at the walls; their half cells enter E by Gauss's law)."""
    rho = rho.astype(np.longdouble)
    if smooth:
        rho = np.concatenate(([rho[0]], 0.25 * (rho[:-2] + 2 * rho[1:-1] + rho[2:]), [rho[-1]]))
    r = np.concatenate(([np.longdouble(0)], np.cumsum(rho[1:-1])))  # R_0 .. R_{N-1}
    slope = (np.sum(r) / n - r) * (dx * dx)
    phi = np.concatenate(([np.longdouble(0)], np.cumsum(slope)))
    phi[-1] = 0
    E = np.empty(n + 1, np.longdouble)
    E[1:-1] = (phi[:-2] - phi[2:]) / (2 * dx)
    E[0] = (phi[0] - phi[1]) / dx - rho[0] * dx / 2
    E[-1] = (phi[-2] - phi[-1]) / dx + rho[-1] * dx / 2
    return phi.astype(np.float64), E.astype(np.float64)


class _Plasma:
    """A plasma of electrons and ions in 64 bits: elastic collisions and charge exchange as
    null collisions; absorbing walls and their field, or periodic in a uniform field."""

    def __init__(self, case, seed, loads, step, cell_units):
        self.n, self.step, self.smooth = case["cells"], step, case.get("smooth", 0)
        self.periodic = case["kind"] == "restart"
        self.E = np.full(self.n + 1, E_EXT)
        self.key = _physics(case, seed)[0].seed
        self.w = DX / case["ppc"]
        self.q, self.m, self.K = (-1.0, 1.0), (1.0, M_ION), (1, case.get("ion_nstep", 1))
        self.sp, self.wall_energy = [], np.zeros((2, 2))
        for k, ld in enumerate(loads):
            vs = 1.0 if cell_units else self.K[k] * DT / DX
            a = [np.asarray(x.cpu() if torch.is_tensor(x) else x)
                 for x in (ld.cell, ld.off, ld.vx, ld.vy, ld.vz, ld.id)]
            s = dict(j=a[0].astype(np.int64), f=a[1].astype(np.float64), id=a[5].astype(np.int64),
                     u=np.stack([x.astype(np.float64) * vs for x in a[2:5]]))
            clock = np.zeros(len(a[0]), np.int64) if ld.state is None else ld.state.astype(np.int64)
            s["due"] = (step + self.K[k]) // self.K[k] - 1 + (clock & 127)  # own steps
            s["pending"] = clock >= 128
            # candidate-free runs of g own steps have probability exp(-g nu K dt)
            s["gap"] = np.floor(np.exp(-np.arange(1, 128) * (NU * self.K[k] * DT)) * 2.0 ** 32)
            self.sp.append(s)
        self.fields()

    def fields(self):
        if self.periodic:
            return
        self.density = np.empty((2, self.n + 1))
        vol = np.full(self.n + 1, DX)
        vol[[0, -1]] = DX / 2
        for k, s in enumerate(self.sp):
            d = np.bincount(s["j"], 1.0 - s["f"], self.n + 1) + \
                np.bincount(s["j"] + 1, s["f"], self.n + 1)
            self.density[k] = self.w * d / vol
        self.phi, self.E = _solve(self.density[1] - self.density[0], self.n, DX, self.smooth)

    def advance(self):
        for k, s in enumerate(self.sp):
            if (self.step + 1) % self.K[k]:
                continue
            own, dt = (self.step + 1) // self.K[k] - 1, self.K[k] * DT
            A = self.q[k] / self.m[k] * (dt * dt / DX) * self.E
            u, j = s["u"], s["j"]
            u[0] += A[j] + s["f"] * (A[j + 1] - A[j])
            x = s["f"] + u[0]
            cross = np.floor(x)
            s["f"] = x - cross
            s["j"] = j = j + cross.astype(np.int64)
            up = s["f"] >= 1.0
            s["f"][up] = 0.0
            j[up] += 1
            if self.periodic:
                j %= self.n
            out = (j < 0) | (j >= self.n)
            if out.any():
                e = 0.5 * self.m[k] * self.w * (DX / dt) ** 2 * (u[:, out] ** 2).sum(0)
                self.wall_energy[k] += e[j[out] < 0].sum(), e[j[out] >= 0].sum()
                for name in ("j", "f", "id", "due", "pending"):
                    s[name] = s[name][~out]
                s["u"] = u[:, ~out]
            due = s["due"] == own
            test = np.nonzero(due & ~s["pending"])[0]
            now = np.nonzero(due & s["pending"])[0]
            to_grid = 127 - own % 127
            if len(test):
                w0 = _philox(s["id"][test], self.step, 0, self.key)[0]
                g = np.minimum(np.searchsorted(-s["gap"], -w0.astype(np.float64), "left"), to_grid)
                s["due"][test] = own + g
                s["pending"][test] = (g > 0) & (g < to_grid)
                now = np.concatenate([now, test[g == 0]])
            if len(now):
                s["due"][now] = own + 1
                s["pending"][now] = False
                self.collide(k, s, now, dt)
        self.step += 1
        self.fields()

    def collide(self, k, s, at, dt):
        r = [_uniform(w) for w in _philox(s["id"][at], self.step, 1 if k == 0 else 2, self.key)]
        if k == 0:  # elastic: a new direction uniform on the sphere, the recoil's energy lost
            c = 1.0 - 2.0 * r[0]
            h = np.sqrt(1.0 - c * c)
            n = np.stack([c, h * np.cos(2 * np.pi * r[1]), h * np.sin(2 * np.pi * r[1])])
            speed = np.sqrt((s["u"][:, at] ** 2).sum(0))
            chi = (s["u"][:, at] * n).sum(0) / np.where(speed > 0, speed, 1.0)
            s["u"][:, at] = speed * np.sqrt(1.0 - 2.0 / M_ION * (1.0 - chi)) * n
        else:  # charge exchange: the velocity of a background neutral (Box-Muller)
            vn = math.sqrt(T_N / M_ION) * dt / DX
            a, b = np.sqrt(-2 * np.log(r[0])), np.sqrt(-2 * np.log(r[2]))
            s["u"][:, at] = vn * np.stack([a * np.cos(2 * np.pi * r[1]),
                                           a * np.sin(2 * np.pi * r[1]),
                                           b * np.cos(2 * np.pi * r[3])])


def exact(case, seed):
    if case["kind"] == "field":
        charge, unit = _deposit(case, seed)
        c = charge.cpu().numpy().astype(object)
        n, z = case["cells"], c[1] - c[0]
        inner = z.copy()
        inner[0] = inner[n] = 0
        R = np.cumsum(inner)
        U = sum(int(n - j) * int(inner[j]) for j in range(n + 1))
        G = np.concatenate(([-2 * U - 2 * n * z[0]], n * (R[:-2] + R[1:-1]) - 2 * U,
                            [2 * n * R[n - 1] - 2 * U + 2 * n * z[n]]))
        lam = DX / case["ppc"] / (2.0 * n * unit)
        return lam * G.astype(np.float64)
    restart = case["kind"] == "restart"
    if not restart and (case["plasma"] != "bounded" or not case["fresh"]):
        return None  # the particle loop of these sizes takes numpy minutes
    if restart:
        p = _Plasma(case, seed, _checkpoint(case, seed), RESTART_STEP, True)
    else:
        gen, device = _generator(seed)
        loads = _particles([(case["ppc"], 1.0), (case["ppc"], 1.0 / math.sqrt(M_ION))],
                           case["cells"], case["precision"], gen, device)
        p = _Plasma(case, seed, loads, 0, False)
    for _ in range(case["steps"]):
        p.advance()
    if restart:
        return [dict(cell=None, off=s["f"], vx=s["u"][0], vy=s["u"][1], vz=s["u"][2], id=None,
                     state=None, yp=np.zeros(len(s["f"]))) for s in p.sp]
    kinetic = [0.5 * p.m[k] * p.w * (DX / (p.K[k] * DT)) ** 2 * (s["u"] ** 2).sum()
               for k, s in enumerate(p.sp)]
    return dict(step=None, live=None, wall_count=None, wall_energy=p.wall_energy, collisions=None,
                kinetic=np.array(kinetic), next_id=None, density=p.density, phi=p.phi, E=p.E)
