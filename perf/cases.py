"""The work that a user of the ECRIS ion time step has it do, as cases that can be timed.

A case is one program of the three forms (a run alone, a batch of runs, a
served request stream) or one call of the allocation-free collision step, with
the sizes, species, meshes and switches of the workloads in
`paper_1507_03392_gb300/inputs.py`, of `bench.py` and of the tests.  Kinds:

  whole    one run from its initial state: load, steps, diagnostics, state out
  advance  a loaded run stepped on, its state read on the device
  sampled  a loaded run stepped one step at a time with its probes sampled
  stream   host arrays in, one step, diagnostics out (new inputs at every pass)
  batch    many runs stepped together, every run's state read on the device
  served   requests submitted to the server and polled until all are done
  collide  one allocation-free collision step on caller-owned arrays

`exact` is the same model in 64 bits with plain torch: positions in metres
instead of fixed point, every particle and every cell at once.
"""
from __future__ import annotations

import ctypes
import math
import time

import numpy as np
import torch

from paper_1507_03392_gb300 import ecris as E
from paper_1507_03392_gb300 import inputs as I

KEYS = ("x", "y", "z", "vx", "vy", "vz")
DEVICE = "cuda"
_stream = None


def stream():
    """The one stream that every run of this file is ordered on, as in one program."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def listed():
    def case(name, kind, n, mesh, steps, **more):
        d = {"name": name, "kind": kind, "species": "Ar", "n": n, "nx": mesh[0], "ny": mesh[1], "nz": mesh[2],
             "steps": steps, "dt": 1e-9, "coulomb": True, "ions": 0.25, "opt_in": False, "runs": 1}
        d.update(more)
        return d

    return [
        # the small plain run in full (1e4 atoms, 1e3 steps): a first look at a source, launch-bound
        case("small_run", "whole", 10_000, (32, 32, 64), 1000, coulomb=False, ions=0.0),
        # an odd, small ensemble with every process on a coarse mesh, as the tests step them
        case("small_collisions", "whole", 20_001, (16, 16, 32), 200, species="O", dt=1e-8, ions=0.5),
        # the paper's own model size (Sec. II): 2e5 macroparticles on 65x65x64 cells, n_e made
        # self-consistent half way
        case("paper_size", "whole", 200_000, (65, 65, 64), 256, dt=1e-8, update_ne=True),
        # the scaled run of the benchmark: 4e6 particles, every process
        case("scaled_run", "advance", 4_000_000, (64, 64, 128), 32),
        # the largest request of the served stream, stepped alone at its time step
        case("largest_run", "whole", 8_000_000, (96, 96, 192), 64, species="Kr", dt=1e-7),
        # the opt-in processes, an on-axis field table and an electric field, without ion-ion collisions
        case("opt_in_run", "advance", 999_999, (32, 32, 64), 64, dt=1e-8, coulomb=False, opt_in=True),
        # exposure images and moments of the plasma: the probes sampled at every step
        case("sampled_run", "sampled", 1_000_000, (32, 32, 64), 16, species="O", dt=1e-8, coulomb=False),
        # end to end: the state from pinned host memory, one step, the diagnostics back
        case("stream_from_host", "stream", 4_000_000, (64, 64, 128), 1),
        # the gas-flow scan: oxygen runs of 2e5 to 2e6 particles in one batch
        case("gas_flow_scan", "batch", 200_000, (32, 32, 64), 32, species="O", coulomb=False, runs=32),
        # the power scan: argon runs of 1e5 to 4e6 particles with collisions between ions in one batch
        case("power_scan", "batch", 100_000, (32, 32, 64), 32, runs=12),
        # a handful of requests of the power scan served together
        case("served_requests", "served", 100_000, (32, 32, 64), 256, runs=6, dt=1e-7),
        # the allocation-free collision step near its limit of 65536 particles
        case("collide_noalloc", "collide", 65_521, (16, 16, 16), 1, dt=1e-8, ions=0.9),
    ]


def draw(rng):
    def lu(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(("whole", "whole", "advance", "advance", "sampled", "stream", "batch", "batch", "collide"))
    mesh = rng.choice(((16, 16, 32), (32, 32, 64), (33, 31, 65), (64, 64, 128), (65, 65, 64), (96, 96, 192)))
    d = {"kind": kind, "species": rng.choice(("Ar", "O", "Kr")), "n": int(lu(1e3, 4e6)) | 1, "nx": mesh[0],
         "ny": mesh[1], "nz": mesh[2], "steps": rng.choice((16, 32, 50, 64)), "dt": lu(1e-9, 1e-7),
         "coulomb": rng.random() < 0.6, "ions": rng.choice((0.0, 0.1, 0.25, 0.5)), "opt_in": rng.random() < 0.2,
         "runs": 1}
    if kind == "sampled":
        d["steps"] = rng.choice((4, 8, 16))
    elif kind == "stream":
        d["steps"] = 1
    elif kind == "batch":
        d.update(runs=rng.randrange(3, 25), n=int(lu(1e3, 5e4)) | 1, nx=32, ny=32, nz=64, steps=rng.choice((16, 32)))
    elif kind == "collide":
        d.update(n=int(lu(100, 65_000)) | 1, nx=rng.randrange(4, 33), ny=rng.randrange(4, 33),
                 nz=rng.randrange(4, 33), steps=1, ions=rng.choice((0.3, 0.9)))
    elif d["n"] * d["steps"] > 1.2e8:
        d["steps"] = 16
    return d


# ---------------------------------------------------------------- inputs


def runs_of(case, seed):
    """(RunParams, particles) of every run of the case: densities, temperatures and sizes drawn as the
    scans of `inputs.py` draw them."""
    rng = np.random.default_rng(seed)
    sizes = np.random.default_rng(977 * case["runs"] + case["n"])   # the sizes belong to the case

    def lu(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    flags = I.F_ALL if case["coulomb"] else I.F_ALL_NO_COULOMB
    more = {}
    if case["opt_in"]:
        flags |= I.F_DOUBLE | I.F_ELASTIC | I.F_RECOMB
        more = {"k3_factor": 0.02, "T_refl_eV": 0.15}
    many = case["runs"] > 1
    out = []
    for i in range(case["runs"]):
        n0 = 3e9 * 100.0 ** (i / max(1, case["runs"] - 1)) if many and not case["coulomb"] else 1e10
        ne, te = (lu(5e10, 2e12), lu(300.0, 3000.0)) if many and case["coulomb"] else (1e11, 1000.0)
        span = 40.0 if case["coulomb"] else 10.0
        n = int(case["n"] * span ** sizes.uniform()) if many else case["n"]
        rp = I.RunParams(species=I.SPECIES[case["species"]], nx=case["nx"], ny=case["ny"], nz=case["nz"], n0_cm3=n0,
                         ne_in_cm3=ne, Te_warm_eV=te, flags=flags, seed=(seed * 1009 + i) % (1 << 40), dt=case["dt"],
                         **more)
        if case["opt_in"]:
            rp.B_axial = I.flat_axial_profile(rp)
        out.append((rp, n))
    return out


def fields_of(case, rp):
    """(E grid, n_e per cell) of a run alone: log-uniform n_e with collisions, as the scaled run has it; a
    synthetic E field with the opt-in processes."""
    if case["runs"] > 1:
        return None, None
    wl = I.Workload("", rp, n=0, steps=0, ne_cells_loguniform=(1e11, 1e12) if case["coulomb"] else None)
    return (I.make_efield(rp, 2e3, -1e3) if case["opt_in"] else None), I.make_ne_cells(wl)


def particles(rp, n, ions, seed):
    """Initial state on the GPU: atoms filling the chamber at T0 (in the zone box when there are no ions),
    ions of Q uniform in 1..8 in the zone box at 0.25 eV."""
    g = torch.Generator(DEVICE).manual_seed(int(seed) % (1 << 62))

    def u():
        return torch.rand(n, generator=g, device=DEVICE)

    ion = u() < ions
    q = torch.randint(1, min(8, rp.species.qmax - 1) + 1, (n,), generator=g, device=DEVICE)
    box = ion if ions > 0 else torch.ones_like(ion)
    r = torch.where(box, 0.018, rp.R0 * (1 - 1e-3)) * u().sqrt()
    th = u() * (2 * math.pi)
    zlo, zhi = torch.where(box, 0.157, rp.L * 1e-3), torch.where(box, 0.213, rp.L * (1 - 1e-3))
    m = rp.species.mass_amu * I.AMU
    sig = torch.where(ion, math.sqrt(0.25 * I.E_CHARGE / m), math.sqrt(rp.T0_eV * I.E_CHARGE / m))
    st = {"x": r * th.cos(), "y": r * th.sin(), "z": zlo + (zhi - zlo) * u()}
    for k in ("vx", "vy", "vz"):
        st[k] = sig * torch.randn(n, generator=g, device=DEVICE)
    st = {k: v.to(torch.float32).contiguous() for k, v in st.items()}
    st["q"] = torch.where(ion, q, 0).to(torch.uint8)
    return st


def empty_state(n):
    out = {k: torch.empty(n, dtype=torch.float32, device=DEVICE) for k in KEYS}
    out["meta"] = torch.empty(n, dtype=torch.int32, device=DEVICE)
    return out


def on_host(st, pinned):
    out = {}
    for k, v in st.items():
        t = torch.empty(v.shape, dtype=v.dtype, pin_memory=pinned)
        t.copy_(v)
        out[k] = t.numpy()
    return out


def probes_of(rp):
    """Every fourth cell of two x-y layers, and screens at the middle and the extraction side (Sec. III.A)."""
    layer = rp.nx * rp.ny
    cells = np.concatenate([np.arange(0, layer, 4) + layer * (rp.nz // 2), np.arange(0, layer, 4) + layer * (rp.nz - 2)])
    return cells.astype(np.uint32), ((0.45 * rp.L, 0.55 * rp.L), (0.9 * rp.L, rp.L))


PIXELS = 64


def prepare(case, seed):
    s = {"case": case, "kind": case["kind"]}
    kind = case["kind"]
    runs = runs_of(case, seed)
    rp, n = runs[0]
    h = stream().cuda_stream
    if kind == "collide":
        return s | collide_inputs(case, seed)
    if kind == "batch":
        b = s["batch"] = E.Batch(stream=h)
        s["handles"] = []
        for i, (rp, n) in enumerate(runs):
            st = particles(rp, n, case["ions"], seed + 31 * i)
            torch.cuda.synchronize()
            s["handles"].append((b.add(rp, st), n))
        s["out"] = empty_state(sum(n for _, n in runs))
    elif kind == "served":
        s["server"] = E.Server(steps_per_tick=32)
        s["requests"] = [(rp, on_host(particles(rp, n, case["ions"], seed + 31 * i), False))
                         for i, (rp, n) in enumerate(runs)]
    else:
        Ef, ne = fields_of(case, rp)
        s["run"] = E.Run(rp, E=Ef, ne_cells=ne, stream=h)
        s["state"] = particles(rp, n, case["ions"], seed)
        s["out"] = empty_state(n)
        torch.cuda.synchronize()
        if kind == "stream":
            s["state"] = on_host(s["state"], True)
        elif kind != "whole":
            s["run"].load(s["state"])
            s["state"] = None
        if kind == "sampled":
            s["run"].set_probes(*probes_of(rp), pixels=PIXELS)
    torch.cuda.synchronize()
    return s


def collide_inputs(case, seed):
    """Caller-owned arrays of the collision step: particles grouped by cell, as a host code keeps them."""
    rp = runs_of(case, seed)[0][0]
    n, nc = case["n"], rp.ncells
    st = particles(rp, n, case["ions"], seed)
    g = torch.Generator(DEVICE).manual_seed(int(seed) + 1)
    cell = torch.randint(0, nc, (n,), generator=g, device=DEVICE).sort().values.to(torch.int32)
    return {"n": n, "cell": cell, "q": st["q"], "v0": [st[k] for k in ("vx", "vy", "vz")],
            "v": [torch.empty_like(st[k]) for k in ("vx", "vy", "vz")],
            "events": torch.zeros(n, dtype=torch.int32, device=DEVICE), "ncells": nc, "rp": rp,
            "vol": 4 * rp.R0 ** 2 * rp.L / nc, "seed": seed % (1 << 40)}


# ---------------------------------------------------------------- one pass


def numbers(d):
    """The diagnostics of a run that are results (a dict of arrays and numbers)."""
    return {k: v for k, v in d.items() if k not in ("steps", "time_s")}


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "collide":
        return run_collide(s)
    if kind == "batch":
        b, out, at = s["batch"], s["out"], 0
        b.step(case["steps"])
        for h, n in s["handles"]:
            ptrs = (ctypes.c_void_p * 6)(*[out[k].data_ptr() + 4 * at for k in KEYS])
            b._check(E.ecris_batch_get_state(b.b, h, ptrs, out["meta"].data_ptr() + 4 * at, 1))
            at += n
        return {"state": out, "diag": numbers(b.diag(s["handles"][-1][0]))}
    if kind == "served":
        srv, steps = s["server"], case["steps"]
        tickets = [srv.submit(rp, st, window_steps=steps, rel_tol=1e-3, min_events=10 ** 15, max_steps=steps)
                   for rp, st in s["requests"]]
        res = [srv.poll(t) for t in tickets]
        while any(r["state"] < E.REQ_DONE for r in res):
            time.sleep(5e-4)
            res = [srv.poll(t) for t in tickets]
        return [{k: r[k] for k in ("state", "steps", "extracted", "lost", "current_A", "power_W")} for r in res]
    r = s["run"]
    if kind == "whole":
        r.load(s["state"])
        if case.get("update_ne"):
            r.step(case["steps"] // 2)
            r.update_ne()
            r.step(case["steps"] - case["steps"] // 2)
        else:
            r.step(case["steps"])
        r.state_to_device(s["out"])
        return {"state": s["out"], "diag": numbers(r.diag(grids=True))}
    if kind == "stream":
        r.load(s["state"])
        r.step(1)
        d = r.diag()
        r.state_to_device(s["out"])
        return {"state": s["out"], "diag": numbers(d)}
    if kind == "sampled":
        for _ in range(case["steps"]):
            r.step(1)
            r.probe_sample()
        r.state_to_device(s["out"])
        return {"state": s["out"], "probes": r.probes()}
    r.step(case["steps"])
    r.state_to_device(s["out"])
    return {"state": s["out"], "diag": numbers(r.diag())}


def run_collide(s):
    # the velocities of this step, as the host code's push left them
    h = stream()
    with torch.cuda.stream(h):
        for v, v0 in zip(s["v"], s["v0"]):
            v.copy_(v0)
        s["events"].zero_()
    rp = s["rp"]
    st = E.ecris_coulomb_collide_noalloc(s["n"], s["cell"].data_ptr(), s["q"].data_ptr(),
                                         *[v.data_ptr() for v in s["v"]], s["events"].data_ptr(), s["ncells"],
                                         rp.species.mass_amu, rp.weight, s["vol"], rp.lnL_ii, rp.dt, s["seed"], 7,
                                         h.cuda_stream, None)
    E.check(None, st)
    return {"vx": s["v"][0], "vy": s["v"][1], "vz": s["v"][2], "events": s["events"]}


def work(case):
    """What a pass cannot do without: each particle's state (28 bytes) in and out once, an ion's once more
    each way in every further step with collisions (its partners are other ions of its cell), and the cell records (16
    bytes) and deposit (8 bytes) once.  Operations: about 120 an atom-step (its random words, move and cell),
    400 an ion-step (with the push, the kick and the events) and 150 for an ion's share of a collision."""
    if case["kind"] == "collide":
        m = case["n"] * case["ions"]
        return {"bytes": case["n"] * 5 + m * 28, "flops": 150.0 * m}
    n = float(sum(k for _, k in runs_of(case, 1)))
    ions, cells = n * case["ions"], case["nx"] * case["ny"] * case["nz"] * case["runs"]
    coll = ions * case["coulomb"]
    b = 56 * n + 24 * cells + 56 * coll * (case["steps"] - 1)
    if case["kind"] == "sampled":
        b += 28 * n * (case["steps"] - 1)   # every sample reads the particles as they are
    return {"bytes": b, "flops": case["steps"] * (120.0 * (n - ions) + 400.0 * ions + 150.0 * coll)}


# ---------------------------------------------------------------- the model in 64 bits

M32 = 0xFFFFFFFF
QE, ME, EPS0 = I.E_CHARGE, 9.1093837015e-31, 8.8541878128e-12
EV_WALL, EV_EXTRACT = 1 << 8, 1 << 9


def philox(pid, c2, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of the counter (pid, 0, c2, 0), key = seed."""
    c0, c1, c2, c3 = pid, torch.zeros_like(pid), torch.full_like(pid, c2), torch.zeros_like(pid)
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def unit(w):
    return ((w >> 8) + 1).double() / 16777216.0


def fires(w, p):
    return w.double() < torch.floor(p * 4294967296.0)


def e1(x):
    """Exponential integral E1 (Abramowitz & Stegun 5.1.11, 5.1.22)."""
    if x <= 1.0:
        s, t = 0.0, 1.0
        for k in range(1, 60):
            t *= -x / k
            s += t / k
        return -0.57721566490153286061 - math.log(x) - s
    f = 0.0
    for k in range(400, 0, -1):
        f = k / (1.0 + k / (x + f))
    return math.exp(-x) / (x + f)


def lotz(p, q, te):
    x = p / te
    return 0.0 if x > 700 else math.sqrt(8 * QE / (math.pi * ME)) * 4.5e-18 * q * e1(x) / (x * te ** 1.5)


def nanbu(s):
    """A of coth A - 1/A = e^-s, by bisection in ln A."""
    y = torch.exp(-s)
    lo, hi = torch.full_like(s, math.log(1e-12)), torch.log(2.0 / -torch.expm1(-s) + 10.0)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        a = torch.exp(mid)
        below = torch.where(a < 1e-3, a / 3 - a ** 3 / 45, 1 / torch.tanh(a) - 1 / a) < y
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    return torch.exp(0.5 * (lo + hi))


def collide_pairs(va, vb, qa, qb, coef, m, dt, w):
    """Nanbu's collision of the pairs (va, vb): [k, 3] velocities, charges, ions of the cell, words of a."""
    g = va - vb
    g2 = (g * g).sum(1)
    gn = g2.sqrt()
    s = coef * (qa * qb) ** 2 * m * dt / gn ** 3
    u = unit(w[1])
    a = nanbu(s.clamp(1e-12, 6.0))
    # below the table's range coth A is 1 to working precision
    a = torch.where(s < 1e-3, 1.0 / -torch.expm1(-s), a)
    cos = torch.where(s > 6.0, 2 * u - 1, 1 + torch.log1p((1 - u) * torch.expm1(-2 * a)) / a).clamp(-1.0, 1.0)
    sin = ((1 - cos) * (1 + cos)).sqrt()
    ph = 2 * math.pi * unit(w[2])
    gp = (g[:, 1] ** 2 + g[:, 2] ** 2).sqrt()
    gx, gy, gz = g.unbind(1)
    h = torch.stack([gp * ph.cos(), -(gx * gy * ph.cos() + gn * gz * ph.sin()) / gp,
                     -(gx * gz * ph.cos() - gn * gy * ph.sin()) / gp], 1)
    flat = torch.stack([torch.zeros_like(gn), gn * ph.cos(), gn * ph.sin()], 1)
    h = torch.where((gp > 0)[:, None], h, flat)
    d = 0.5 * (h * sin[:, None] - g * (1 - cos)[:, None])
    d = torch.where((g2 > 0)[:, None], d, 0.0)
    return va + d, vb - d


def collisions(v, pid, cell, q, ncells, coef, dt, seed, step):
    """Takizawa-Abe pairs of every cell's ions in the order of (word 0 of stream 1, id); v: [k, 3], in place."""
    w0 = philox(pid, 4 * step + 1, seed)[0]
    order = torch.sort(cell * (1 << 32) + w0, stable=True).indices
    count = torch.bincount(cell, minlength=ncells)
    first = torch.cumsum(count, 0) - count
    c = cell[order]
    m, rank = count[c], torch.arange(len(c), device=c.device) - first[c]
    pairs = torch.where(m % 2 == 0, rank % 2 == 0, (rank >= 3) & (rank % 2 == 1)).logical_and(m > 1)
    trips = (m % 2 == 1) & (m >= 3) & (rank == 0)
    qd = q.double()

    def one(ia, ib, mm, t):
        v[ia], v[ib] = collide_pairs(v[ia], v[ib], qd[ia], qd[ib], coef, mm, t, philox(pid[ia], 4 * step + 1, seed))

    at = pairs.nonzero()[:, 0]
    one(order[at], order[at + 1], m[at].double(), dt)
    at = trips.nonzero()[:, 0]
    a, b, c3 = order[at], order[at + 1], order[at + 2]
    for i, j in ((a, b), (b, c3), (c3, a)):
        one(i, j, m[at].double(), 0.5 * dt)
    return order[(pairs | trips).nonzero()[:, 0]], m


def coulomb_coef(rp, vol):
    mu = 0.5 * rp.species.mass_amu * I.AMU
    return rp.lnL_ii / (4 * math.pi) * (QE * QE / (EPS0 * mu)) ** 2 * rp.weight / vol


class Model:
    """One run in 64 bits."""

    def __init__(self, rp, st, Ef, ne_cells):
        self.rp, self.step_no = rp, 0
        self.m = rp.species.mass_amu * I.AMU
        self.p = torch.stack([st[k].double() for k in KEYS[:3]], 1)
        self.v = torch.stack([st[k].double() for k in KEYS[3:]], 1)
        self.q = st["q"].long()
        self.pid = torch.arange(len(self.q), device=DEVICE)
        self.d = (2 * rp.R0 / rp.nx, 2 * rp.R0 / rp.ny, rp.L / rp.nz)
        self.zm = rp.L / (1 + math.sqrt((rp.B_ext - rp.B_min) / (rp.B_inj - rp.B_min)))
        if rp.B_axial is not None:
            self.spline()
        ix, iy, iz = (torch.arange(k, device=DEVICE) + 0.5 for k in (rp.nx, rp.ny, rp.nz))
        c = torch.cartesian_prod(iz * self.d[2], iy * self.d[1] - rp.R0, ix * self.d[0] - rp.R0)
        self.bmag = self.field(c.flip(1).double()).norm(dim=1)
        self.zone = (self.bmag < rp.B_ecr).long()
        ins = torch.full_like(self.bmag, rp.ne_in_cm3) if ne_cells is None else torch.from_numpy(ne_cells).to(DEVICE).double()
        self.te = torch.tensor([rp.Te_cold_eV, rp.Te_warm_eV], device=DEVICE, dtype=torch.float64)
        self.set_ne(1e6 * torch.where(self.zone == 1, ins, rp.ne_out_cm3))
        self.ef = None if Ef is None else torch.from_numpy(Ef).to(DEVICE).double()
        self.rates()
        self.charge, self.since = torch.zeros_like(self.bmag), 0

    def spline(self):
        """Second derivatives of the natural cubic spline through the on-axis samples."""
        y = np.asarray(self.rp.B_axial, dtype=np.float64)
        n, h = len(y), self.rp.L / (len(y) - 1)
        a = np.diag(np.full(n - 2, 4.0)) + np.diag(np.ones(n - 3), 1) + np.diag(np.ones(n - 3), -1)
        m = np.zeros(n)
        m[1:-1] = np.linalg.solve(a, 6 * (y[2:] - 2 * y[1:-1] + y[:-2]) / h ** 2)
        self.ax = [torch.from_numpy(k).to(DEVICE) for k in (y, m)] + [h]

    def field(self, p):
        rp, (x, y, z) = self.rp, p.unbind(1)
        if rp.B_axial is not None:
            ya, ma, h = self.ax
            k = (z / h).long().clamp(0, len(ya) - 2)
            t = z / h - k
            u = 1 - t
            y0, y1, m0, m1 = ya[k], ya[k + 1], ma[k], ma[k + 1]
            b0 = u * y0 + t * y1 + h * h / 6 * ((u ** 3 - u) * m0 + (t ** 3 - t) * m1)
            b1 = (y1 - y0) / h + h / 6 * ((3 * t * t - 1) * m1 - (3 * u * u - 1) * m0)
            b2 = u * m0 + t * m1
        else:
            left = z <= self.zm
            a = torch.where(left, 0.5 * (rp.B_inj - rp.B_min), -0.5 * (rp.B_ext - rp.B_min))
            k = torch.where(left, math.pi / self.zm, math.pi / (rp.L - self.zm))
            ph = k * torch.where(left, z, z - self.zm)
            b0 = rp.B_min + torch.where(left, a * (1 + ph.cos()), a * (ph.cos() - 1))
            b1, b2 = -a * k * ph.sin(), -a * k * k * ph.cos()
        hc = rp.B_hex / rp.R0 ** 2
        return torch.stack([-0.5 * x * b1 + hc * 2 * x * y, -0.5 * y * b1 + hc * (x * x - y * y),
                            b0 - 0.25 * (x * x + y * y) * b2], 1)

    def efield(self, p):
        """Trilinear between cell centres, clamped at the faces."""
        rp = self.rp
        lo, f = [], []
        for k, (n, o) in enumerate(((rp.nx, rp.R0), (rp.ny, rp.R0), (rp.nz, 0.0))):
            g = ((p[:, k] + o) / self.d[k] - 0.5).clamp(0, n - 1)
            i = g.long().clamp(0, n - 2)
            lo.append(i)
            f.append(g - i)
        out = 0.0
        for c in range(8):
            b = (c & 1, c >> 1 & 1, c >> 2)
            w = torch.ones_like(f[0])
            for k in range(3):
                w = w * (f[k] if b[k] else 1 - f[k])
            out = out + w[:, None] * self.ef[((lo[2] + b[2]) * rp.ny + lo[1] + b[1]) * rp.nx + lo[0] + b[0]]
        return out

    def set_ne(self, ne):
        """n_e (m^-3) of every cell and the delta of the printed 3x3 stencil."""
        rp = self.rp
        self.ne = ne
        g = torch.nn.functional.pad(ne.view(rp.nz, 1, rp.ny, rp.nx), (1, 1, 1, 1), mode="replicate")[:, 0]

        def at(dy, dx):
            return g[:, 1 + dy:1 + dy + rp.ny, 1 + dx:1 + dx + rp.nx].reshape(-1)

        sx = at(-1, 0) - at(1, 0) + 0.5 * (at(-1, 1) + at(-1, -1) - at(1, -1) - at(1, 1))
        sy = at(0, 1) - at(0, -1) + 0.5 * (at(1, 1) + at(-1, 1) - at(1, -1) - at(-1, -1))
        rl = torch.where(ne > 0, 2.38e-6 * self.te[self.zone].sqrt() / (self.bmag * self.d[0]) / ne, 0.0)
        self.delta = torch.stack([-rl * sx, -rl * sy, torch.zeros_like(rl)], 1)

    def rates(self):
        """k1, k2, k3, kr by zone and Q (m^3/s): Lotz, its multiples, and Seaton's recombination."""
        rp = self.rp
        ip, nout = rp.species.ladder()
        qm = rp.species.qmax
        k = np.zeros((4, 2, qm + 1))
        for zone, te in enumerate((rp.Te_cold_eV, rp.Te_warm_eV)):
            for q in range(qm):
                k[0, zone, q] = lotz(ip[q], nout[q], te)
                if rp.flags & I.F_DOUBLE and q + 1 < qm:
                    k[1, zone, q] = rp.k2_factor * lotz(ip[q] + ip[q + 1], nout[q], te)
                if rp.flags & I.F_DOUBLE and q + 2 < qm and rp.k3_factor > 0:
                    k[2, zone, q] = rp.k3_factor * lotz(ip[q] + ip[q + 1] + ip[q + 2], nout[q], te)
            for q in range(1, qm + 1):
                if rp.flags & I.F_RECOMB:
                    lam = 157890.0 * q * q / (te * 11604.518)
                    k[3, zone, q] = 5.197e-20 * q * math.sqrt(lam) * (0.4288 + 0.5 * math.log(lam) + 0.469 * lam ** (-1 / 3))
        self.k = torch.from_numpy(k).to(DEVICE)

    def cell_of(self, p):
        rp = self.rp
        i = [((p[:, k] + o) / self.d[k]).long().clamp(0, n - 1)
             for k, (n, o) in enumerate(((rp.nx, rp.R0), (rp.ny, rp.R0), (rp.nz, 0.0)))]
        return (i[2] * rp.ny + i[1]) * rp.nx + i[0]

    def thermal(self, u, sigma):
        """Two Box-Muller pairs of the four words: (x, y, z)."""
        r1, r2 = ((-2 * unit(u[k]).log()).sqrt() * sigma for k in (0, 2))
        t1, t2 = 2 * math.pi * unit(u[1]), 2 * math.pi * unit(u[3])
        return torch.stack([r1 * t1.cos(), r1 * t1.sin(), r2 * t2.cos()], 1)

    def step(self):
        rp, v, dt, qm = self.rp, self.v, self.rp.dt, self.rp.species.qmax
        fl, c2 = rp.flags, 4 * self.step_no
        sig0 = math.sqrt(rp.T0_eV * QE / self.m)
        # Boris push of the ions
        i = (self.q > 0).nonzero()[:, 0]
        if len(i):
            h = (self.q[i].double() * (QE / self.m) * 0.5 * dt)[:, None]
            e = 0.0 if self.ef is None else h * self.efield(self.p[i])
            t = h * self.field(self.p[i])
            m = v[i] + e
            m = m + torch.linalg.cross(m + torch.linalg.cross(m, t), 2 * t / (1 + (t * t).sum(1, keepdim=True)))
            v[i] = m + e
        old = self.p
        new = old + v * dt
        r2 = new[:, 0] ** 2 + new[:, 1] ** 2
        out = (r2 > rp.R0 ** 2) | (new[:, 2] < 0) | (new[:, 2] >= rp.L)
        self.p = new
        if out.any():
            self.leave(out.nonzero()[:, 0], old, new, sig0, c2)
        # collisions with electrons and atoms, in the cell of the new position
        cell = self.cell_of(self.p)
        zone, ne, stay = self.zone[cell], self.ne[cell], ~out
        w = philox(self.pid, c2, rp.seed)
        k = self.k[:, zone, self.q]
        tot = k.sum(0)
        p = -torch.expm1(-ne * tot * dt)
        hit = fires(w[0], p) & stay & (tot > 0)
        if hit.any():
            j = hit.nonzero()[:, 0]
            share = torch.cumsum(k[:, j], 0) / tot[j] * p[j]
            up = torch.where(fires(w[0][j], share[0]), 1,
                             torch.where(fires(w[0][j], share[1]), 2, torch.where(fires(w[0][j], share[2]), 3, -1)))
            self.q[j] += up
        i = (stay & (self.q >= 1)).nonzero()[:, 0]
        if len(i):
            q = self.q[i]
            vrel = ((v[i] ** 2).sum(1) + 8 * rp.T0_eV * QE / (math.pi * self.m)).sqrt()
            n0 = rp.n0_cm3 * 1e6
            cx = torch.where(q != 2, n0 * rp.sigma1_cm2 * 1e-4 * q.double(), 0.0)
            el = n0 * rp.sigma_el1_cm2 * 1e-4 * q.double() if fl & I.F_ELASTIC else torch.zeros_like(cx)
            pt = -torch.expm1(-(cx + el) * vrel * dt)
            hit = fires(w[1][i], pt)
            is_cx = hit & fires(w[1][i], pt * torch.where(cx + el > 0, cx / (cx + el), 0.0))
            a = i[hit & ~is_cx]
            if len(a):
                atom = self.thermal(philox(self.pid[a], c2 + 3, rp.seed), sig0)
                d = philox(self.pid[a], c2 + 2, rp.seed)
                g = (v[a] - atom).norm(dim=1, keepdim=True)
                v[a] = 0.5 * (v[a] + atom) + 0.5 * g * self.direction(d[0], d[1])
            a = i[is_cx & (q == 1)]
            if len(a):
                v[a] = self.thermal(philox(self.pid[a], c2 + 3, rp.seed), sig0)
            a = i[is_cx & (q >= 3)]
            if len(a):
                u = philox(self.pid[a], c2 + 3, rp.seed)
                v[a] += math.sqrt(rp.E_cx_eV * QE / self.m) * self.direction(u[0], u[1])
                self.q[a] -= 1
            # heating kick
            te = self.te[zone[i]]
            d2 = 3.715e-6 * rp.lnL_ei * dt / (rp.species.mass_amu ** 2 * te.sqrt()) * ne[i] * self.q[i].double() ** rp.ei_charge_power
            n = self.direction(w[2][i], w[3][i]) + self.delta[cell[i]]
            nn = n.norm(dim=1, keepdim=True)
            v[i] += torch.where(nn > 0, d2.sqrt()[:, None] * n / nn, 0.0)
            if fl & I.F_COULOMB:
                vv = v[i]
                collisions(vv, self.pid[i], cell[i], self.q[i], rp.ncells, coulomb_coef(rp, math.prod(self.d)), dt,
                           rp.seed, self.step_no)
                v[i] = vv
        self.charge += torch.bincount(cell, weights=self.q.double(), minlength=rp.ncells)
        self.step_no += 1
        self.since += 1

    def direction(self, a, b):
        c = 2 * unit(a) - 1
        s, t = (1 - c * c).clamp(min=0).sqrt(), 2 * math.pi * unit(b)
        return torch.stack([s * t.cos(), s * t.sin(), c], 1)

    def leave(self, i, old, new, sig0, c2):
        """Wall hits and extraction: the first crossing of the segment, and the re-emission (cosine law)."""
        rp, (o, d) = self.rp, (old[i], new[i] - old[i])
        inf = torch.full((len(i),), math.inf, dtype=torch.float64, device=DEVICE)
        a, b = (d[:, :2] ** 2).sum(1), (o[:, :2] * d[:, :2]).sum(1)
        c = (o[:, :2] ** 2).sum(1) - rp.R0 ** 2
        den = b + (b * b - a * c).clamp(min=0).sqrt()
        fr = torch.where((new[i, :2] ** 2).sum(1) > rp.R0 ** 2, torch.where(den > 0, -c / den, 0.0).clamp(min=0), inf)
        f0 = torch.where(new[i, 2] < 0, -o[:, 2] / d[:, 2], inf)
        fl = torch.where(new[i, 2] >= rp.L, (rp.L - o[:, 2]) / d[:, 2], inf)
        f, kind = torch.stack([fr, f0, fl]).min(0)
        x = o + f[:, None] * d
        rc = (x[:, :2] ** 2).sum(1).sqrt()
        gone = (kind == 2) & (rc < rp.r_ap)
        u = philox(self.pid[i], c2 + 2, rp.seed)
        refl = math.sqrt(rp.T_refl_eV * QE / self.m) if rp.T_refl_eV > 0 else sig0
        sig = torch.where(gone | (self.q[i] == 0), sig0, refl)
        vn, rt = ((-2 * unit(u[k]).log()).sqrt() * sig for k in (0, 1))
        t1, t2 = rt * (2 * math.pi * unit(u[2])).cos(), rt * (2 * math.pi * unit(u[2])).sin()
        eps = 1e-6 * rp.L
        ux, uy = x[:, 0] / rc, x[:, 1] / rc
        side = torch.stack([-vn * ux - t1 * uy, -vn * uy + t1 * ux, t2], 1)
        sgn = torch.where((kind == 2) & ~gone, -1.0, 1.0)
        flat = torch.stack([t1, t2, sgn * vn], 1)
        self.v[i] = torch.where((kind == 0)[:, None], side, flat)
        wall = torch.stack([(rp.R0 - eps) * ux, (rp.R0 - eps) * uy, x[:, 2]], 1)
        plane = torch.stack([x[:, 0], x[:, 1], torch.where(kind == 2, rp.L - eps, eps)], 1)
        at = torch.where((kind == 0)[:, None], wall, plane)
        inlet = torch.tensor(rp.inlet, dtype=torch.float64, device=DEVICE)
        self.p[i] = torch.where(gone[:, None], inlet, at)
        self.q[i] = 0

    def update_ne(self):
        self.set_ne(self.rp.weight * self.charge / (self.since * math.prod(self.d)))
        self.charge.zero_()
        self.since = 0


def exact(case, seed):
    runs = runs_of(case, seed)
    kind = case["kind"]
    if kind == "served":
        return None   # counts, and currents that are counts times constants
    if kind != "collide" and case["coulomb"] and case["steps"] * case["dt"] > 1e-7:
        # with collisions an ion that rounding puts into the next cell pairs both cells anew, and from there
        # on their ions are another sample of the same process: no particle has a value that it ought to have
        return None
    if kind == "collide":
        s = collide_inputs(case, seed)
        v = torch.stack([k.double() for k in s["v0"]], 1)
        i = (s["q"] > 0).nonzero()[:, 0]
        vv = v[i]
        collisions(vv, i, s["cell"][i].long(), s["q"][i].long(), s["ncells"], coulomb_coef(s["rp"], s["vol"]),
                   s["rp"].dt, s["seed"], 7)
        v[i] = vv
        return {"vx": v[:, 0], "vy": v[:, 1], "vz": v[:, 2], "events": None}
    done = []
    for i, (rp, n) in enumerate(runs):
        Ef, ne = fields_of(case, rp)
        m = Model(rp, particles(rp, n, case["ions"], seed + 31 * i), Ef, ne)
        sums = None
        if kind == "sampled":
            cells = torch.from_numpy(probes_of(rp)[0].astype(np.int64)).to(DEVICE)
            slot = torch.full((rp.ncells,), -1, device=DEVICE)
            slot[cells] = torch.arange(len(cells), device=DEVICE)
            qs = rp.species.qmax + 1
            sums = torch.zeros(len(cells) * qs, 7, dtype=torch.float64, device=DEVICE)
        for k in range(case["steps"]):
            m.step()
            if case.get("update_ne") and k + 1 == case["steps"] // 2:
                m.update_ne()
            if sums is not None:
                at = slot[m.cell_of(m.p)]
                j = (at >= 0).nonzero()[:, 0]
                rows = torch.cat([torch.ones(len(j), 1, device=DEVICE, dtype=torch.float64), m.v[j], m.v[j] ** 2], 1)
                sums.index_add_(0, at[j] * qs + m.q[j], rows)
        done.append(torch.cat([m.p, m.v], 1))
        del m
    all_ = torch.cat(done)
    out = {"state": {k: all_[:, j] for j, k in enumerate(KEYS)} | {"meta": None}}
    if kind == "sampled":
        out["probes"] = {"samples": None, "moments": sums.view(len(cells), qs, 7), "screens": None}
    return out
