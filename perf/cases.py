"""The work a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values.  Kinds:
  run       one simulation handle, stepped some steps, then its state read back
  batch     many independent foils stepped together (a parameter scan), fields of every run read back
  whole     one run from host arrays to its results: create, upload, step, read back, destroy
  readout   the read-outs of a finished run: both spectra and the energy record
  snapshot  the skin-layer snapshot with its per-particle values
  electron  single electrons in plane waves (leapfrog or RK4)
  hist      the spectrum of momenta that the caller holds on the device

Fields and momenta are single-precision numbers in the library (the C ABI only
widens them), so a program keeps them in single precision, as run() does here.
"""
import math

import numpy as np
import torch

import paper_1008_1685_gb300 as picrr
from paper_1008_1685_gb300.binding import spectrum_noalloc

PROTON = 1836.15267343  # proton mass / electron mass
MEC2 = 0.51099895000    # electron rest energy, MeV
CFL, LAMBDA_UM, SOURCE = 0.95, 0.8, 8
FIELDS = (picrr.EX, picrr.EY, picrr.EZ, picrr.BY, picrr.BZ)
WAVE_CASES = 3


def _run(name, cells, cpl, n, slab0, slab, ne, a0, pol, rr, te, ti, shapes, steps, particles):
    return dict(name=name, kind="run", cells=cells, cpl=cpl, n=n, slab0=slab0, slab=slab, ne=ne, a0=a0, pol=pol, rr=rr,
                te=te, ti=ti, unit=shapes[0], interval=shapes[1], slots=shapes[2], steps=steps, particles=particles)


def listed():
    plain = (4096, 8, 2)  # the library's default launch shapes
    return [
        # a program that looks at the whole state after every step, on a test-sized box (5 lambda at lambda/100)
        _run("one_step", 500, 100.0, 1000, 30, 400, 5.0, 30.0, 0, True, 0.5, 0.01, plain, 1, True),
        # the small single run (20 lambda at lambda/200, 64 per cell and species, LP a0 = 200): launches count
        _run("small_run", 4000, 200.0, 12_800, 60, 200, 64.0, 200.0, 0, True, 0.2, 0.001, plain, 48, True),
        # the paper-scale run (60 lambda at lambda/1000, 400 per cell and species) with the default shapes
        _run("paper_run", 60_000, 1000.0, 400_000, 100, 1000, 90.0, 350.0, 1, True, 0.1, 0.001, plain, 192, False),
        # the large single run (100 lambda at lambda/2000, 64M particles) with the shapes the tuner picks for it
        _run("large_run", 200_000, 2000.0, 32_000_000, 100, 4000, 100.0, 500.0, 1, True, 0.1, 0.001, (16384, 96, 4), 96,
             False),
        # late phase of a run: hot electrons spread thinly over the whole box, odd sizes
        _run("thin_plasma", 700_001, 500.0, 4_100_003, 999, 698_000, 0.06, 100.0, 1, True, 20.0, 0.05, plain, 192, False),
        # part of the 256-run scan (15,000 cells each, drawn thickness, density, ppc, polarization, RR) in its shapes
        dict(name="scan_batch", kind="batch", runs=48, cells=15_000, cpl=500.0, ppc_lo=32, ppc_hi=256, th_lo=0.5, th_hi=2.0,
             unit=8192, interval=96, slots=2, steps=192),
        # one run of a request stream through the single-run API, from host arrays to its state on the host
        dict(name="whole_run", kind="whole", cells=15_000, cpl=500.0, n=100_000, slab0=60, slab=500, ne=80.0, a0=300.0,
             pol=0, rr=True, te=0.1, ti=0.001, unit=4096, interval=64, slots=2, steps=128, ordered=True),
        # what is read when a large run ends: ion and electron spectra (200 bins of 0..2000 MeV) and the energies
        dict(name="read_out", kind="readout", cells=200_000, cpl=2000.0, n=8_000_000, bins=200, e_max=2000.0, te=300.0,
             ti=0.3),
        # the skin-layer snapshot of a paper-scale run: d and chi of every electron
        dict(name="snapshot", kind="snapshot", cells=60_000, cpl=1000.0, n=400_000, te=200.0),
        # the paper's single-electron accuracy test as a scan: RK4 of the lab-frame LL equation with its derivative term
        dict(name="electron_rk4", kind="electron", n=4096, rk4=True, rr=True, deriv=True, dt=0.01, steps=2000, every=100),
        # and the leapfrog pusher over more electrons, fewer rows kept
        dict(name="electron_leapfrog", kind="electron", n=20_000, rk4=False, rr=True, deriv=False, dt=0.01, steps=1000,
             every=500),
        # the spectrum without device allocation, from momenta that the caller holds on the device
        dict(name="device_spectrum", kind="hist", n=16_000_000, bins=200, e_max=2000.0, p=500.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: single runs twice as often as the others."""
    kind = rng.choice(["run", "run", "run", "batch", "whole", "readout", "snapshot", "electron", "hist"])
    if kind == "run":
        thin = rng.random() < 0.4
        n = _log(rng, 800, 16_000_000 if not thin else 5_000_000)
        if thin:  # 2 to 12 particles per cell, hot, over nearly the whole box
            slab = max(64, int(n / rng.uniform(2.0, 12.0)))
            slab0, te, ne = rng.randint(12, 900), rng.uniform(5.0, 30.0), rng.uniform(0.02, 0.1)
            cells = slab0 + slab + rng.randint(20, 900)
            cpl = 500.0
        else:     # a foil of 50 to 8000 particles per cell and the pulse in front of it
            slab = max(50, int(n / min(8000.0, 50.0 * (n / 800.0) ** 0.5)))
            slab0, te, ne = rng.randint(20, 200), rng.uniform(0.05, 0.2), rng.uniform(30.0, 100.0)
            cells = slab0 + slab + _log(rng, 300, 190_000)
            cpl = 200.0 if n <= 30_000 else rng.choice([500.0, 1000.0, 2000.0])
        if n < 4_000_000 or thin:
            shapes = rng.choice([(4096, 8, 2), (4096, 16, 2), (8192, 96, 2), (4096, 64, 2)])
        else:
            shapes = rng.choice([(16384, 96, 4), (4096, 8, 2), (8192, 32, 4)])
        steps = rng.choice([1, 24, 40, 48]) if n <= 30_000 else rng.choice([64, 96, 101])
        c = _run("", cells, cpl, n, slab0, slab, ne, rng.uniform(50.0, 300.0), rng.randint(0, 1), rng.random() < 0.7, te,
                 0.05 if thin else 0.001, shapes, steps, n <= 30_000)
        del c["name"]
        return c
    if kind == "batch":
        return dict(kind="batch", runs=_log(rng, 2, 48), cells=rng.randint(3000, 15_000), cpl=500.0, ppc_lo=rng.randint(8, 32),
                    ppc_hi=rng.randint(64, 256), th_lo=rng.uniform(0.2, 0.5), th_hi=rng.uniform(0.8, 2.0),
                    unit=rng.choice([4096, 8192]), interval=rng.choice([8, 64, 96]), slots=2, steps=rng.choice([96, 128, 192]))
    if kind == "whole":
        n = _log(rng, 10_000, 1_000_000)
        return dict(kind="whole", cells=rng.randint(8000, 30_000), cpl=500.0, n=n, slab0=rng.randint(30, 100),
                    slab=rng.randint(250, 1000), ne=rng.uniform(30.0, 150.0), a0=rng.uniform(100.0, 600.0),
                    pol=rng.randint(0, 1), rr=rng.random() < 0.5, te=0.1, ti=0.001, unit=4096, interval=rng.choice([8, 64]),
                    slots=2, steps=128, ordered=rng.random() < 0.6)
    if kind == "readout":
        return dict(kind="readout", cells=rng.randint(4000, 200_000), cpl=1000.0, n=_log(rng, 10_000, 8_000_000),
                    bins=_log(rng, 20, 20_000), e_max=rng.uniform(500.0, 3000.0), te=rng.uniform(1.0, 500.0),
                    ti=rng.uniform(0.05, 0.5))
    if kind == "snapshot":
        return dict(kind="snapshot", cells=rng.randint(4000, 100_000), cpl=1000.0, n=_log(rng, 10_000, 1_000_000),
                    te=rng.uniform(1.0, 300.0))
    if kind == "electron":
        rk4 = rng.random() < 0.5
        rr = rng.random() < 0.8
        return dict(kind="electron", n=_log(rng, 16, 20_000), rk4=rk4, rr=rr, deriv=rk4 and rng.random() < 0.5, dt=0.01,
                    steps=rng.randint(200, 1000), every=rng.choice([20, 50, 100]))
    return dict(kind="hist", n=_log(rng, 10_000, 16_000_000), bins=_log(rng, 20, 65_000), e_max=rng.uniform(500.0, 3000.0),
                p=rng.uniform(1.0, 800.0))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _plasma(case, seed):
    """A thermal plasma slab: cells (int32, in order), offsets shared by both species, momenta of each (float32)."""
    g = torch.Generator(device="cuda").manual_seed(1 + int(seed))
    n, slab = case["n"], case.get("slab", case["cells"] - 200)
    if n % slab == 0:  # the same number in every cell, as a foil is loaded
        cell = torch.arange(slab, device="cuda", dtype=torch.int32).repeat_interleave(n // slab)
    else:
        cell = torch.randint(0, slab, (n,), generator=g, device="cuda", dtype=torch.int32).sort().values
    cell = cell + case.get("slab0", 100)
    off = torch.rand(n, generator=g, device="cuda")
    p = [[torch.randn(n, generator=g, device="cuda") * t for _ in range(3)] for t in (case["te"], case.get("ti", 0.0))]
    return cell, off, p


def _host(v):
    return v.cpu().numpy()


def _smooth_fields(case, seed):
    """A laser-like wave over a slowly varying longitudinal field, on the grid of the case."""
    r = np.random.default_rng(1000 + int(seed))
    nx, dx = case["cells"], 2 * math.pi / case["cpl"]
    a, k, ph = r.uniform(100.0, 300.0), r.uniform(0.8, 1.2), r.uniform(0.0, 6.28)
    node, half = np.arange(nx + 1) * dx, (np.arange(nx) + 0.5) * dx
    f = [0.3 * a * np.sin(0.2 * k * half + ph), a * np.sin(k * node + ph), 0.5 * a * np.cos(k * node + ph),
         -0.5 * a * np.cos(k * half + ph), a * np.sin(k * half + ph)]
    return [np.float32(x).astype(np.float64) for x in f]


def _weight(case):
    return case["ne"] * case["slab"] / case["n"]


def _open(case, host):
    s = picrr.Sim(case["cells"] / case["cpl"], case["cpl"], cfl=CFL, lambda_um=LAMBDA_UM, rr_on=case["rr"],
                  sort_interval=case["interval"], source_node=SOURCE)
    cell, off, p = host
    s.load_particles_f32(picrr.ELECTRON, cell, off, *p[0], _weight(case), -1.0, 1.0)
    s.load_particles_f32(picrr.ION, cell, off, *p[1], _weight(case), 1.0, PROTON)
    s.inject_laser(case["a0"], case["pol"], picrr.ENV_SIN2, 10.0)
    s.set_shapes(case["unit"], case["interval"], case["slots"])
    return s


def _scan(case, seed):
    """The runs of a scan, each drawn as the library's benchmark draws them, the foil close to the source."""
    r = np.random.default_rng(50_000 + int(seed))
    return [dict(x0=float(r.uniform(0.08, 0.16)), th=float(r.uniform(case["th_lo"], case["th_hi"])), ne=float(r.uniform(30.0, 150.0)),
                 a0=float(r.uniform(100.0, 600.0)), pol=int(r.integers(0, 2)), rr=bool(r.integers(0, 2)),
                 ppc=int(r.integers(case["ppc_lo"], case["ppc_hi"] + 1)), seed=int(r.integers(1, 1 << 40))) for _ in range(case["runs"])]


def _electrons(case, seed):
    r = np.random.default_rng(90_000 + int(seed))
    return [dict(wave=i % WAVE_CASES, a0=float(r.uniform(20.0, 350.0)), tau=float(r.uniform(30.0, 60.0)), x0=float(r.uniform(-1.0, 1.0)),
                 p0=(float(r.uniform(-200.0, 10.0)), float(r.uniform(-5.0, 5.0)), float(r.uniform(-5.0, 5.0)))) for i in range(case["n"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("run", "whole"):
        cell, off, p = _plasma(case, seed)
        host = [_host(cell), _host(off), [[_host(x) for x in q] for q in p]]
        if kind == "run":
            return dict(case=case, sim=_open(case, host))
        if not case["ordered"]:  # a restart from particles as they are read back: not in cell order
            at = np.random.default_rng(7 + int(seed)).permutation(case["n"])
            host = [host[0][at], host[1][at], [[x[at] for x in q] for q in host[2]]]
        pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()  # noqa: E731
        return dict(case=case, host=[pin(host[0]), pin(host[1]), [[pin(x) for x in q] for q in host[2]]])
    if kind == "batch":
        b = picrr.Batch(case["cpl"], max_runs=case["runs"], cfl=CFL, lambda_um=LAMBDA_UM, sort_interval=case["interval"])
        b.set_shapes(case["unit"], case["interval"], case["slots"])
        ids = [b.add_run(case["cells"] / case["cpl"], d["x0"], d["th"], d["ne"], d["a0"], d["pol"], 10.0, 10**12, rr_on=d["rr"],
                         ppc=d["ppc"], seed=d["seed"], source_node=SOURCE) for d in _scan(case, seed)]
        return dict(case=case, batch=b, ids=ids)
    if kind in ("readout", "snapshot"):
        cell, off, p = _plasma(case, seed)
        s = picrr.Sim(case["cells"] / case["cpl"], case["cpl"], cfl=CFL, lambda_um=LAMBDA_UM, source_node=SOURCE)
        s.set_fields(*_smooth_fields(case, seed))
        cell, off = _host(cell), _host(off)
        s.load_particles_f32(picrr.ELECTRON, cell, off, *map(_host, p[0]), 0.01, -1.0, 1.0)
        if kind == "readout":
            s.load_particles_f32(picrr.ION, cell, off, *map(_host, p[1]), 0.01, 1.0, PROTON)
        return dict(case=case, sim=s)
    if kind == "electron":
        return dict(case=case, electrons=_electrons(case, seed))
    g = torch.Generator(device="cuda").manual_seed(3 + int(seed))
    p = [torch.randn(case["n"], generator=g, device="cuda") * case["p"] for _ in range(3)]
    return dict(case=case, p=p, counts=torch.empty(case["bins"], dtype=torch.float64, device="cuda"))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _state_of(sim, with_particles):
    out = {"f%d" % c: np.float32(sim.field(c)) for c in FIELDS}
    if with_particles:
        for sp in (picrr.ELECTRON, picrr.ION):
            q = sim.particles(sp)
            for k in ("x", "px", "py", "pz"):
                out["s%d_%s" % (sp, k)] = np.float32(q[k])
            out["s%d_flag" % sp] = q["flag"]
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "run":
        state["sim"].step(case["steps"])
        return _state_of(state["sim"], case["particles"])
    if kind == "whole":
        s = _open(case, state["host"])
        s.step(case["steps"])
        out = _state_of(s, True)
        s.close()
        return out
    if kind == "batch":
        b = state["batch"]
        b.step(case["steps"])
        return [np.stack([np.float32(b.field(r, c)) for r in state["ids"]]) for c in FIELDS]
    if kind == "readout":
        s = state["sim"]
        ion, _ = s.spectra(picrr.ION, case["bins"], 0.0, case["e_max"])
        el, radiated = s.spectra(picrr.ELECTRON, case["bins"], 0.0, case["e_max"])
        return dict(ion=ion, el=el, energy=s.energy(), radiated=np.float64(radiated))
    if kind == "snapshot":
        d = state["sim"].snapshot(picrr.ELECTRON, chi_flag=0.1)
        return dict(x=d["x"], px=d["px"], pperp=d["pperp"], d=np.float32(d["d"]), chi=np.float32(d["chi"]),
                    d_max=np.float32(d["d_max"]), chi_max=np.float32(d["chi_max"]), n_flagged=d["n_flagged"])
    if kind == "electron":
        return picrr.electron_scan(state["electrons"], integrator=picrr.INTEGRATOR_RK4 if case["rk4"] else picrr.INTEGRATOR_LEAPFROG,
                                   rr=case["rr"], deriv=case["deriv"], dt=case["dt"], nsteps=case["steps"], every=case["every"])
    p = state["p"]
    rc, why = spectrum_noalloc(p[0].data_ptr(), p[1].data_ptr(), p[2].data_ptr(), case["n"], 1.0, 0.01, case["bins"], 0.0,
                               case["e_max"], state["counts"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    if rc:
        raise RuntimeError(why)
    return state["counts"]


def work(case):
    """Bytes and operations a pass cannot do without: each step reads and writes every particle (cell, offset, three
    momenta: 40 bytes) and the five fields (40 bytes a node); about 200 operations a particle and step."""
    kind = case["kind"]
    if kind in ("run", "whole", "batch"):
        if kind == "batch":
            n = case["runs"] * (case["ppc_lo"] + case["ppc_hi"]) * round((case["th_lo"] + case["th_hi"]) / 2 * case["cpl"])
            nodes = case["runs"] * case["cells"]
        else:
            n, nodes = 2 * case["n"], case["cells"]
        read = 20 * nodes + (24 * n if kind == "whole" or case.get("particles") else 0)
        load = 40 * n if kind == "whole" else 0  # the caller's arrays up, the device copy written
        return {"bytes": case["steps"] * (40 * n + 40 * nodes) + read + load, "flops": case["steps"] * (200 * n + 30 * nodes)}
    if kind == "readout":  # momenta of both species, for the spectra and the energies, and the fields
        return {"bytes": 2 * 2 * 12 * case["n"] + 20 * case["cells"] + 16 * case["bins"], "flops": 2 * 2 * 15 * case["n"]}
    if kind == "snapshot":
        return {"bytes": 24 * case["n"] + 40 * case["n"] + 20 * case["cells"], "flops": 80 * case["n"]}
    if kind == "electron":
        rows = case["n"] * (case["steps"] // case["every"])
        return {"bytes": 64 * case["n"] + 40 * rows, "flops": case["n"] * case["steps"] * (4 * 110 if case["rk4"] else 110)}
    return {"bytes": 12 * case["n"] + 8 * case["bins"], "flops": 15 * case["n"]}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _incident(run, t):
    """(Ey, Ez) of the pulse at retarded time t."""
    tau = run["tau"]
    if t < 0.0 or t > tau:
        return 0.0, 0.0
    g = math.sin(math.pi * t / tau) ** 2
    if run["pol"] == picrr.LP:
        return run["a0"] * g * math.sin(t), 0.0
    a = run["a0"] / math.sqrt(2.0)
    return a * g * math.sin(t), -a * g * math.cos(t)


def _pic(runs, nx, cpl, steps):
    """Plain 1D PIC of several runs on equal grids.  A run: tau, a0, pol, rr, and species as (cell, off, px, py, pz,
    weight, charge, mass).  Returns the fields [Ex, Ey, Ez, By, Bz] and the species' tensors (x in cells)."""
    f8 = dict(dtype=torch.float64, device="cuda")
    B, dx = len(runs), 2 * math.pi / cpl
    dt, eps = CFL * dx, (4.0 / 3.0) * math.pi * 2.8179403262e-9 / LAMBDA_UM
    W, pad = nx + 4, 2  # node or half node i of run b at b * W + pad + i
    Ex, Ey, Ez, By, Bz = (torch.zeros(B, W, **f8) for _ in range(5))
    parts = []
    for sp in (0, 1):
        arrs = [torch.cat([r["species"][sp][k].to(torch.float64 if k else torch.int64) for r in runs]) for k in range(5)]
        ns = [len(r["species"][sp][0]) for r in runs]
        per = lambda v: torch.tensor(v, **f8).repeat_interleave(torch.tensor(ns, device="cuda"))  # noqa: E731
        base = torch.arange(B, device="cuda").repeat_interleave(torch.tensor(ns, device="cuda")) * W + pad
        parts.append(dict(cell=arrs[0], off=arrs[1], p=arrs[2:], base=base, live=torch.ones(len(base), dtype=torch.bool, device="cuda"),
                          qw=per([r["species"][sp][5] * r["species"][sp][6] for r in runs]), qm=per([r["species"][sp][6] / r["species"][sp][7] for r in runs]),
                          rr=per([float(r["rr"] and sp == 0) for r in runs]), some_rr=any(r["rr"] for r in runs) and sp == 0))
    lanes = 16  # spread the adds of a dense cell over several rows
    for step in range(steps):
        J = torch.zeros(3, lanes, B * W, **f8)
        fl = [F.reshape(-1) for F in (Ex, Ey, Ez, By, Bz)]
        for s in parts:
            c, f, base = s["cell"], s["off"], s["base"]
            px, py, pz = s["p"]
            q = base + c.clamp(max=nx - 1)
            h = (f < 0.5).long()
            jb, g = q - h, f - 0.5 + h
            at = lambda F, i, w: F[i] * (1 - w) + F[i + 1] * w  # noqa: E731
            ey, ez, ex = at(fl[1], q, f), at(fl[2], q, f), at(fl[0], jb, g)
            by, bz = at(fl[3], jb, g), at(fl[4], jb, g)
            k = 0.5 * dt * s["qm"]
            mx, my, mz = px + k * ex, py + k * ey, pz + k * ez
            ig = 1 / torch.sqrt(1 + mx * mx + my * my + mz * mz)
            ty, tz = k * by * ig, k * bz * ig
            sf = 2 / (1 + ty * ty + tz * tz)
            ux, uy, uz = mx + my * tz - mz * ty, my - mx * tz, mz + mx * ty
            lx, ly, lz = mx + sf * (uy * tz - uz * ty) + k * ex, my - sf * ux * tz + k * ey, mz + sf * ux * ty + k * ez
            if s["some_rr"]:
                ax, ay, az = 0.5 * (lx + px), 0.5 * (ly + py), 0.5 * (lz + pz)
                igb = 1 / torch.sqrt(1 + ax * ax + ay * ay + az * az)
                vx, vy, vz = ax * igb, ay * igb, az * igb
                fx, fy, fz = -(ex + vy * bz - vz * by), -(ey - vx * bz), -(ez + vx * by)
                ve = vx * ex + vy * ey + vz * ez
                br = fx * fx + fy * fy + fz * fz + (ay * fz - az * fy) ** 2 + (az * fx - ax * fz) ** 2 + (ax * fy - ay * fx) ** 2
                e = -eps * dt * s["rr"]
                lx, ly, lz = lx + e * (fy * bz - fz * by - ve * ex + br * vx), ly + e * (-fx * bz - ve * ey + br * vy), lz + e * (fx * by - ve * ez + br * vz)
            live = s["live"]
            px, py, pz = (torch.where(live, a, b) for a, b in ((lx, px), (ly, py), (lz, pz)))
            ign = 1 / torch.sqrt(1 + px * px + py * py + pz * pz)
            x1 = c + f + torch.where(live, CFL * px * ign, torch.zeros_like(px))
            gone = (x1 < 0) | (x1 >= nx)
            x1 = x1.clamp(0.0, float(nx))
            c1 = torch.where(live, x1.floor().long(), c)
            f1 = torch.where(live, x1 - c1, f)
            lane = torch.arange(len(c), device="cuda") % lanes * (B * W) + base
            qw = s["qw"] * live
            for cc, ff in ((c, f), (c1, f1)):  # the time-averaged linear shape
                for comp, v in ((1, py), (2, pz)):
                    cur = 0.5 * qw * v * ign
                    J[comp].view(-1).index_add_(0, lane + cc, cur * (1 - ff))
                    J[comp].view(-1).index_add_(0, lane + cc + 1, cur * ff)
            a = torch.minimum(c, c1)  # charge that crossed half nodes a and a + 1
            one = torch.ones_like(f)
            o0, n0 = torch.where(c == a, 1 - f, 0 * f), torch.where(c1 == a, 1 - f1, 0 * f)
            o1, n1 = torch.where(c == a, one, 1 - f), torch.where(c1 == a, one, 1 - f1)
            J[0].view(-1).index_add_(0, lane + a, qw / CFL * (o0 - n0))
            J[0].view(-1).index_add_(0, lane + a + 1, qw / CFL * (o1 - n1))
            s["cell"], s["off"], s["p"], s["live"] = c1, f1, [px, py, pz], live & ~gone
        Jx, Jy, Jz = (j.view(B, W) for j in J.sum(1))
        inc = torch.tensor([[v for t in (step * dt, step * dt + 0.5 * dt + 0.5 * dx, (step + 1) * dt) for v in _incident(r, t)] for r in runs], **f8)
        i0, hc = pad, 0.5 * CFL
        hn, nd = slice(i0, i0 + nx), slice(i0, i0 + nx + 1)  # half nodes, nodes

        def half_b(ay, az):
            By[:, hn] += hc * (Ez[:, i0 + 1:i0 + nx + 1] - Ez[:, hn])
            Bz[:, hn] -= hc * (Ey[:, i0 + 1:i0 + nx + 1] - Ey[:, hn])
            Bz[:, i0 + SOURCE - 1] += hc * ay
            By[:, i0 + SOURCE - 1] -= hc * az

        half_b(inc[:, 0], inc[:, 1])
        oy, oz = Ey.clone(), Ez.clone()
        inner = slice(i0 + 1, i0 + nx)
        Ey[:, inner] += -CFL * (Bz[:, inner] - Bz[:, i0:i0 + nx - 1]) - dt * Jy[:, inner]
        Ez[:, inner] += CFL * (By[:, inner] - By[:, i0:i0 + nx - 1]) - dt * Jz[:, inner]
        Ey[:, i0 + SOURCE] += CFL * inc[:, 2]
        Ez[:, i0 + SOURCE] += CFL * inc[:, 3]
        km = (CFL - 1) / (CFL + 1)
        for E, o in ((Ey, oy), (Ez, oz)):
            E[:, i0] = o[:, i0 + 1] + km * (E[:, i0 + 1] - o[:, i0])
            E[:, i0 + nx] = o[:, i0 + nx - 1] + km * (E[:, i0 + nx - 1] - o[:, i0 + nx])
        half_b(inc[:, 4], inc[:, 5])
        Ex[:, hn] -= dt * Jx[:, hn]
    return [F[:, hn if k in (0, 3, 4) else nd] for k, F in enumerate((Ex, Ey, Ez, By, Bz))], parts


def _foil_offsets(seed, c0, ncell, ppc):
    """SplitMix64 outputs (Steele, Lea and Flood 2014) of the foil's macro-particles, as 24-bit offsets."""
    n = (np.arange(c0 * ppc, (c0 + ncell) * ppc, dtype=np.uint64) + np.uint64(1))
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + n * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(40)).astype(np.float64) / 16777216.0


def _kinetic(p):
    p2 = sum(x.astype(np.float64) ** 2 for x in p)
    return p2 / (np.sqrt(1.0 + p2) + 1.0)


def _counts(e, bins, e_max, unit):
    k = np.floor(e / e_max * bins)
    return np.bincount(k[k < bins].astype(np.int64), minlength=bins) * (unit / (e_max / bins))


def _wave(kind, a0, tau, phi):
    """Ey, Ez and their derivatives by the phase, for the three waves."""
    s, c = np.sin(phi), np.cos(phi)
    a = a0 * math.sqrt(0.5)
    on = (phi >= 0) & (phi <= tau)
    se, ce = np.sin(np.pi * phi / tau), np.cos(np.pi * phi / tau)
    g, dg = se * se, 2 * se * ce * np.pi / tau
    pick = lambda x, y, z: np.where(kind == 0, x, np.where(kind == 1, y, np.where(on, z, 0.0)))  # noqa: E731
    return pick(a0 * c, a * c, a0 * g * c), pick(0, a * s, 0), pick(-a0 * s, -a * s, a0 * (dg * c - g * s)), pick(0, a * c, 0)


def _exact_electrons(case, seed):
    el = _electrons(case, seed)
    kind = np.array([e["wave"] for e in el])
    a0, tau, x = (np.array([e[k] for e in el]) for k in ("a0", "tau", "x0"))
    p = np.array([e["p0"] for e in el]).T.copy()
    dt, eps = case["dt"], (4.0 / 3.0) * math.pi * 2.8179403262e-9 / LAMBDA_UM
    rows = []

    def force(phi, p):
        g = np.sqrt(1 + (p * p).sum(0))
        vx, vy, vz = p / g
        ey, ez, dey, dez = _wave(kind, a0, tau, phi)
        lx, ly, lz = vy * ey + vz * ez, ey * (1 - vx), ez * (1 - vx)
        f = [-lx, -ly, -lz]
        if case["rr"]:
            ve = vy * ey + vz * ez
            sq = g * g * (lx * lx + ly * ly + lz * lz - ve * ve)
            f = [f[0] + eps * (ly * ey + lz * ez - sq * vx), f[1] + eps * (-lx * ey + ve * ey - sq * vy), f[2] + eps * (-lx * ez + ve * ez - sq * vz)]
            if case["deriv"]:
                k = eps * g * (1 - vx)
                f = [f[0] - k * (vy * dey + vz * dez), f[1] - k * dey * (1 - vx), f[2] - k * dez * (1 - vx)]
        return np.array(f), vx

    for s in range(case["steps"]):
        t = s * dt
        if case["rk4"]:
            f1, v1 = force(t - x, p)
            f2, v2 = force(t + 0.5 * dt - (x + 0.5 * dt * v1), p + 0.5 * dt * f1)
            f3, v3 = force(t + 0.5 * dt - (x + 0.5 * dt * v2), p + 0.5 * dt * f2)
            f4, v4 = force(t + dt - (x + dt * v3), p + dt * f3)
            x = x + dt / 6 * (v1 + 2 * v2 + 2 * v3 + v4)
            p = p + dt / 6 * (f1 + 2 * f2 + 2 * f3 + f4)
        else:
            ey, ez, _, _ = _wave(kind, a0, tau, t - x)
            h = -0.5 * dt
            mx, my, mz = p[0], p[1] + h * ey, p[2] + h * ez
            gm = np.sqrt(1 + mx * mx + my * my + mz * mz)
            ty, tz = -h * ez / gm, h * ey / gm
            sf = 2 / (1 + ty * ty + tz * tz)
            ux, uy, uz = mx + my * tz - mz * ty, my - mx * tz, mz + mx * ty
            L = np.array([mx + sf * (uy * tz - uz * ty), my - sf * ux * tz + h * ey, mz + sf * ux * ty + h * ez])
            if case["rr"]:
                q = 0.5 * (L + p)
                g = np.sqrt(1 + (q * q).sum(0))
                vx, vy, vz = q / g
                fx, fy, fz = -(vy * ey + vz * ez), -ey * (1 - vx), -ez * (1 - vx)
                ve = vy * ey + vz * ez
                sq = g * g * (fx * fx + fy * fy + fz * fz - ve * ve)
                L = L - dt * eps * np.array([fy * ey + fz * ez + sq * vx, -fx * ey - ve * ey + sq * vy, -fx * ez - ve * ez + sq * vz])
            p = L
            x = x + dt * p[0] / np.sqrt(1 + (p * p).sum(0))
        if (s + 1) % case["every"] == 0:
            rows.append(np.stack([np.full(len(x), (s + 1) * dt), x, *p], 1))
    return np.stack(rows, 1)


def exact(case, seed):
    kind, dx = case["kind"], 2 * math.pi / case.get("cpl", 1.0)
    if kind == "electron":
        return _exact_electrons(case, seed) if case["n"] * case["steps"] * (4 if case["rk4"] else 1) <= 60_000_000 else None
    if kind == "hist":
        g = torch.Generator(device="cuda").manual_seed(3 + int(seed))
        e = MEC2 * _kinetic([_host(torch.randn(case["n"], generator=g, device="cuda") * case["p"]) for _ in range(3)])
        return _counts(e, case["bins"], case["e_max"], 0.01)
    if kind == "batch":
        runs = []
        for d in _scan(case, seed):
            c0, nc = round(d["x0"] * case["cpl"]), round(d["th"] * case["cpl"])
            n = nc * d["ppc"]
            cell = torch.arange(c0, c0 + nc, device="cuda").repeat_interleave(d["ppc"])
            off = torch.from_numpy(_foil_offsets(d["seed"], c0, nc, d["ppc"])).cuda()
            z = torch.zeros(n, device="cuda", dtype=torch.float64)
            runs.append(dict(tau=10.0 * 2 * math.pi, a0=d["a0"], pol=d["pol"], rr=d["rr"],
                             species=[(cell, off, z, z, z, d["ne"] / d["ppc"], -1.0, 1.0), (cell, off, z, z, z, d["ne"] / d["ppc"], 1.0, PROTON)]))
        if sum(len(r["species"][0][0]) for r in runs) * case["steps"] > 1_000_000_000:
            return None
        return [F.cpu() for F in _pic(runs, case["cells"], case["cpl"], case["steps"])[0]]
    if kind in ("run", "whole"):
        if case["n"] * case["steps"] > 1_000_000_000:
            return None
        cell, off, p = _plasma(case, seed)
        if kind == "whole" and not case["ordered"]:
            at = torch.from_numpy(np.random.default_rng(7 + int(seed)).permutation(case["n"])).cuda()
            cell, off, p = cell[at], off[at], [[x[at] for x in q] for q in p]
        w = _weight(case)
        one = dict(tau=10.0 * 2 * math.pi, a0=case["a0"], pol=case["pol"], rr=case["rr"],
                   species=[(cell, off, *p[0], w, -1.0, 1.0), (cell, off, *p[1], w, 1.0, PROTON)])
        F, parts = _pic([one], case["cells"], case["cpl"], case["steps"])
        out = {"f%d" % c: F[c][0].cpu() for c in FIELDS}
        if kind == "whole" or case["particles"]:
            for sp, s in enumerate(parts):
                out["s%d_x" % sp] = ((s["cell"] + s["off"]) * dx).cpu()
                for k, v in zip(("px", "py", "pz"), s["p"]):
                    out["s%d_%s" % (sp, k)] = v.cpu()
                out["s%d_flag" % sp] = None
        return out
    cell, off, p = _plasma(case, seed)
    F = _smooth_fields(case, seed)
    if kind == "readout":
        f = [[_host(x) for x in q] for q in p]
        ke, ki = _kinetic(f[0]), _kinetic(f[1])
        a, b = SOURCE + 1, case["cells"] - 1  # accounting region: nodes a..b, half nodes a..b-1, every half node for Ex
        hc = 0.5 * CFL
        dy, dz = hc * np.diff(F[2])[a:b], hc * np.diff(F[1])[a:b]
        uf = 0.5 * ((F[1][a:b + 1] ** 2).sum() + (F[2][a:b + 1] ** 2).sum() + (F[3][a:b] ** 2 - dy ** 2).sum() + (F[4][a:b] ** 2 - dz ** 2).sum() + (F[0] ** 2).sum())
        energy = np.array([uf * dx, ke.sum() * 0.01 * dx, ki.sum() * 0.01 * dx * PROTON, 0.0, 0.0, 0.0])
        return dict(ion=_counts(ki * MEC2 * PROTON, case["bins"], case["e_max"], 0.01 * dx), el=_counts(ke * MEC2, case["bins"], case["e_max"], 0.01 * dx),
                    energy=energy, radiated=None)
    cell, f = _host(cell).astype(np.int64), _host(off).astype(np.float64)
    px, py, pz = (_host(x).astype(np.float64) for x in p[0])
    node = lambda A: A[cell] * (1 - f) + A[cell + 1] * f  # noqa: E731
    jb = cell - (f < 0.5)
    g = f - 0.5 + (f < 0.5)
    half = lambda A: A[jb] * (1 - g) + A[jb + 1] * g  # noqa: E731
    ex, ey, ez, by, bz = half(F[0]), node(F[1]), node(F[2]), half(F[3]), half(F[4])
    ga = np.sqrt(1 + px * px + py * py + pz * pz)
    vx, vy, vz = px / ga, py / ga, pz / ga
    fx, fy, fz = -(ex + vy * bz - vz * by), -(ey - vx * bz), -(ez + vx * by)
    br = fx * fx + fy * fy + fz * fz + (py * fz - pz * fy) ** 2 + (pz * fx - px * fz) ** 2 + (px * fy - py * fx) ** 2
    d = (4.0 / 3.0) * math.pi * 2.8179403262e-9 / LAMBDA_UM * br
    chi = np.sqrt(br) * 2 * math.pi * 3.8615926796e-7 / LAMBDA_UM
    return dict(x=(cell + f) * dx, px=px, pperp=np.sqrt(py * py + pz * pz), d=d, chi=chi, d_max=np.array(d.max()),
                chi_max=np.array(chi.max()), n_flagged=None)
