"""The work that users of this library have it do, as cases to be measured.

A pass of a `run` case is what a user's program does for one simulation: open it from a
configuration, advance it, read the energies and the state back, close it.  A `batch` case
does that for many small simulations advanced together, a `restore` case goes on from a
checkpoint held on the host, and a `diag` case takes the diagnostics of a simulation that is
open.  All go through the C-ABI binding `paper_2310_11393_gb300.pic`.

The pulse crosses its focus (or enters the slab) within the steps of a case, so that the
electrons are hot and evaluate the whole incident field, as they do around the focus of the
long runs.  Outputs of single-precision runs are returned in single precision, the electrons
in the order of their ids (an electron that left the box: a row of zeros).

`exact` advances the same inputs with plain torch operations in 64 bits: order-2 shapes, the
closed-form incident fields, the momentum updates, Esirkepov's current and the Yee scheme with
first-order Mur faces, written from the paper's formulas.
"""
import math

import numpy as np
import torch

from paper_2310_11393_gb300 import pic

TWO_PI = 2.0 * math.pi
BEAMS = {"plane": pic.PIC_BEAM_PLANE, "lp": pic.PIC_BEAM_LP, "rp": pic.PIC_BEAM_RP, "gauss2d": pic.PIC_BEAM_GAUSS2D}
PUSHERS = {"boris": pic.PIC_PUSHER_BORIS, "vay": pic.PIC_PUSHER_VAY, "hc": pic.PIC_PUSHER_HC}

# What every case says, with the values that most of them have.
DEFAULTS = {
    "kind": "run", "dim": 2, "nx": 64, "ny": 1, "nz": 1, "cells": 32, "precision": "fp32", "beam": "lp", "a0": 10.0,
    "waist": 1.0, "s": 27.1, "duration": 14.7, "gauss_envelope": False, "focus_step": 25, "ref_cell": 0.0,
    "slab_lo": 0.25, "slab_hi": 0.75, "slab_margin": 0, "n_e": 0.01, "ppc": 4, "supergauss": False, "pusher": "boris",
    "incident_grid": False, "sort_every": 0, "tile_x": 0, "tile_y": 0, "tile_z": 0, "chunk": 0, "steps": 50,
    "members": 1, "particles": True, "fields": True,
}


def listed():
    return [
        # the 1D plane-wave preset in double precision while its pulse is in the slab: 32 768 electrons,
        # many short steps
        {"name": "1d_plane_fp64", "dim": 1, "nx": 4096, "cells": 64, "precision": "fp64", "beam": "plane", "a0": 1.0,
         "duration": 23.55, "ref_cell": 700.0, "ppc": 16, "steps": 1000},
        # a small 1D run in single precision at an odd size: latency and launches
        {"name": "1d_plane_odd", "dim": 1, "nx": 1531, "cells": 64, "beam": "plane", "a0": 3.0, "duration": 23.55,
         "gauss_envelope": True, "focus_step": 500, "pusher": "vay", "slab_lo": 0.3, "slab_hi": 0.9, "ppc": 5,
         "steps": 700},
        # the smallest run: a short 2D simulation, opened, stepped, read and closed
        {"name": "2d_lp_small", "nx": 96, "ny": 80, "waist": 0.5, "n_e": 0.05, "slab_lo": 0.17, "slab_hi": 0.85,
         "steps": 50},
        # the 2D benchmark workload around its focus (tile and work item as measured for it)
        {"name": "2d_lp_1024", "nx": 1024, "ny": 1024, "n_e": 0.05, "ppc": 8, "focus_step": 150, "tile_x": 32,
         "tile_y": 16, "chunk": 1024, "steps": 300, "fields": False},
        # the 2D Gaussian beam in a dense super-Gaussian slab, with the default tile
        {"name": "2d_gauss_2048", "nx": 2048, "ny": 1024, "beam": "gauss2d", "a0": 4.86, "waist": 16.0,
         "duration": TWO_PI, "n_e": 0.31, "ppc": 4, "supergauss": True, "slab_lo": 0.08, "slab_hi": 0.62,
         "slab_margin": 4, "focus_step": 75, "steps": 150, "particles": False},
        # a 2D run in double precision
        {"name": "2d_rp_fp64", "nx": 256, "ny": 256, "precision": "fp64", "beam": "rp", "a0": 20.0, "waist": 0.7,
         "ppc": 8, "focus_step": 50, "steps": 100},
        # the 3D benchmark workload around its focus, the largest: 16.8 M electrons, 33.5 M cells
        {"name": "3d_rp_512", "dim": 3, "nx": 512, "ny": 256, "nz": 256, "cells": 24, "beam": "rp", "a0": 20.0,
         "waist": 0.7, "focus_step": 75, "tile_x": 16, "tile_y": 8, "tile_z": 4, "chunk": 4096, "steps": 150,
         "fields": False},
        # a 3D request of the served stream's kind, default tile
        {"name": "3d_rp_160", "dim": 3, "nx": 160, "ny": 160, "nz": 160, "cells": 24, "beam": "rp", "a0": 20.0,
         "waist": 0.7, "focus_step": 50, "steps": 100, "fields": False},
        # a small 3D run at odd sizes with a linearly polarised pulse and the Higuera-Cary update
        {"name": "3d_lp_odd", "dim": 3, "nx": 75, "ny": 61, "nz": 53, "cells": 24, "waist": 0.6, "ppc": 3,
         "pusher": "hc", "focus_step": 30, "steps": 60},
        # uneven 2D simulations advanced together
        {"name": "2d_batch", "kind": "batch", "members": 12, "nx": 384, "ny": 384, "n_e": 0.02, "ppc": 8,
         "focus_step": 60, "steps": 120},
        # a checkpoint restored from the host, advanced and read back
        {"name": "2d_restore", "kind": "restore", "nx": 512, "ny": 512, "beam": "rp", "a0": 20.0, "waist": 0.7,
         "focus_step": 60, "ppc": 4, "steps": 20},
        # the energies and the energy-angle histogram of a running 3D simulation
        {"name": "3d_diag", "kind": "diag", "dim": 3, "nx": 256, "ny": 128, "nz": 128, "cells": 24, "beam": "rp",
         "a0": 20.0, "waist": 0.7, "focus_step": 60, "steps": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: 1D, 2D or 3D runs (half of all), batches, restores, diagnostics."""
    c = {"kind": rng.choice(["run", "run", "run", "run", "run", "batch", "restore", "diag"])}
    c["dim"] = {"run": rng.choice([1, 2, 2, 3, 3]), "batch": 2, "restore": rng.choice([2, 3]),
                "diag": rng.choice([2, 3])}[c["kind"]]
    d = c["dim"]
    top = {1: 6000, 2: 1024, 3: 224}[d] if c["kind"] == "run" else {1: 6000, 2: 512, 3: 128}[d]
    low = {1: 256, 2: 64, 3: 40}[d]
    n = _log_int(rng, low, top)
    c["nx"] = n
    c["ny"] = max(40, int(n * rng.uniform(0.6, 1.1))) if d > 1 else 1
    c["nz"] = max(40, int(n * rng.uniform(0.6, 1.1))) if d > 2 else 1
    c["cells"] = {1: 64, 2: 32, 3: 24}[d]
    c["precision"] = "fp64" if rng.random() < (0.5 if d == 1 else 0.15) else "fp32"
    c["beam"] = "plane" if d == 1 else rng.choice(["lp", "rp", "rp"] if d == 3 else ["lp", "lp", "rp", "gauss2d"])
    c["a0"] = round(math.exp(rng.uniform(0.0, math.log(20.0))), 3)
    c["waist"] = round(rng.uniform(4.0, 16.0) if c["beam"] == "gauss2d" else rng.uniform(0.5, 2.0), 3)
    c["duration"] = 23.55 if d == 1 else TWO_PI
    c["gauss_envelope"] = d == 1 and rng.random() < 0.5
    c["ppc"] = rng.randint(1, 16 if d < 3 else 6)
    c["n_e"] = round(math.exp(rng.uniform(math.log(0.001), math.log(0.05))), 5)
    c["pusher"] = rng.choice(["boris", "boris", "boris", "vay", "hc"])
    c["slab_lo"], c["slab_hi"] = round(rng.uniform(0.15, 0.3), 3), round(rng.uniform(0.6, 0.85), 3)
    if c["kind"] == "run":
        c["incident_grid"] = rng.random() < 0.1
        c["sort_every"] = rng.choice([0, 0, 0, 0, 0, 10])
        if d > 1 and rng.random() < 0.5:
            tiles = [(32, 16, 1), (64, 8, 1), (16, 8, 1)] if d == 2 else [(16, 8, 4), (8, 8, 4), (16, 8, 8)]
            c["tile_x"], c["tile_y"], c["tile_z"] = rng.choice(tiles)
            c["chunk"] = rng.choice([1024, 2048, 4096])
    if c["precision"] == "fp64" and d == 3:
        c["tile_x"], c["tile_y"], c["tile_z"], c["chunk"] = 0, 0, 0, 0
    if c["kind"] == "batch":
        c["members"] = rng.randint(3, 12)
    # steps such that a case stays well below the largest listed one, and electrons meet the pulse
    most = {1: 800, 2: 160, 3: 80}[d]
    per_step = _electrons(_full(c)) * c.get("members", 1) * (40 if c["precision"] == "fp64" else 1)
    c["steps"] = 0 if c["kind"] == "diag" else 20 if c["kind"] == "restore" else max(20, min(most, int(4e8 / (per_step + 1))))
    c["focus_step"] = max(10, c["steps"] // 2)
    c["fields"] = c["nx"] * c["ny"] * c["nz"] < 1_500_000
    return c


def _full(case):
    return {**DEFAULTS, **case}


def _slab(c):
    n = (c["nx"], c["ny"], c["nz"])
    lo, hi = [], []
    for d in range(c["dim"]):
        if d > 0 and c["slab_margin"]:
            lo.append(c["slab_margin"])
            hi.append(n[d] - c["slab_margin"])
        else:
            lo.append(max(4, int(n[d] * c["slab_lo"])))
            hi.append(min(n[d] - 4, int(n[d] * c["slab_hi"])))
    return lo + [0] * (3 - c["dim"]), hi + [1] * (3 - c["dim"])


def _electrons(c):
    lo, hi = _slab(c)
    return c["ppc"] * math.prod(hi[d] - lo[d] for d in range(c["dim"]))


def _members(case, seed):
    """Physical parameters of each simulation of a case; the seed sets phases, amplitudes and positions."""
    c = _full(case)
    rng = np.random.default_rng([int(seed), 2310])
    out = []
    for k in range(c["members"]):
        m = dict(c)
        if c["members"] > 1:      # uneven sizes (from a third of the largest up), both beams
            f = 1.0 if k == 0 else (1.0 + 2.0 * ((k * 7) % c["members"]) / c["members"]) / 3.0
            m["nx"] = m["ny"] = max(48, int(c["nx"] * f))
            m["beam"] = c["beam"] if k % 2 == 0 else "rp"
            m["ppc"] = 1 + (c["ppc"] + 3 * k) % 12
        m["a0"] = c["a0"] * float(rng.uniform(0.95, 1.0))
        m["phi0"] = float(rng.uniform(-1.0, 1.0))
        m["seed"] = int(rng.integers(1, 2**62))
        dim = m["dim"]
        dx = TWO_PI / m["cells"]
        m["dx"], m["dt"] = dx, 0.95 * dx / math.sqrt(dim)
        m["n"] = (m["nx"], m["ny"] if dim > 1 else 1, m["nz"] if dim > 2 else 1)
        m["focus"] = tuple(0.5 * m["n"][d] * dx if d < dim else 0.0 for d in range(3))
        m["t_focus"] = m["focus_step"] * m["dt"]
        m["w0"] = m["waist"] * TWO_PI
        m["a"] = m["psi0"] = 0.0
        if m["beam"] == "plane":
            m["focus"] = (m["ref_cell"] * dx, 0.0, 0.0)
        elif m["beam"] in ("lp", "rp"):
            m["a"] = math.sqrt((1.0 + 0.5 * m["w0"] ** 2) ** 2 - 1.0)      # k^2 w0^2 = 2 (sqrt(1 + (ka)^2) - 1)
            m["psi0"] = m["a0"] / _focal_peak(m)
        lo, hi = _slab(m)
        m["lo"], m["hi"] = lo, hi
        m["prof"] = (0.5 * (lo[0] + hi[0]) * dx, 0.8 * (hi[0] - lo[0]) * dx, 0.0)     # centre, FWHM, cut
        out.append(m)
    return out


def _config(m):
    cfg = pic.pic_config()
    cfg.dim, cfg.dx, cfg.dt, cfg.cfl = m["dim"], m["dx"], m["dt"], 0.95
    cfg.precision = pic.PIC_FP64 if m["precision"] == "fp64" else pic.PIC_FP32
    cfg.beam = BEAMS[m["beam"]]
    cfg.envelope = pic.PIC_ENV_GAUSS if m["gauss_envelope"] else pic.PIC_ENV_SIN2
    cfg.a0, cfg.duration, cfg.w0, cfg.phi0, cfg.t_focus = m["a0"], m["duration"], m["w0"], m["phi0"], m["t_focus"]
    cfg.a_param, cfg.s_param, cfg.psi0 = m["a"], m["s"], m["psi0"]
    for d in range(3):
        cfg.n[d], cfg.focus[d], cfg.slab_lo[d], cfg.slab_hi[d] = m["n"][d], m["focus"][d], m["lo"][d], m["hi"][d]
        cfg.tile[d] = (m["tile_x"], m["tile_y"], m["tile_z"])[d] if d < m["dim"] else 0
    cfg.n_e, cfg.ppc, cfg.seed, cfg.chunk = m["n_e"], m["ppc"], m["seed"], m["chunk"]
    cfg.pusher, cfg.incident_grid, cfg.sort_every = PUSHERS[m["pusher"]], int(m["incident_grid"]), m["sort_every"]
    if m["supergauss"]:
        cfg.profile, cfg.prof_order = pic.PIC_PROFILE_SUPERGAUSS, 12
        cfg.prof_x0, cfg.prof_fwhm, cfg.prof_cut = m["prof"]
    return cfg


# ---- what a user's program does -----------------------------------------------------------
def prepare(case, seed):
    members = _members(case, seed)
    state = {"members": members, "configs": [_config(m) for m in members], "allocator": _allocator(),
             "stream": torch.cuda.current_stream().cuda_stream}
    m = members[0]
    # the host buffers that the program reads the state into (the binding's arrays are their views)
    if m["kind"] != "diag" and m["particles"]:
        state["records"] = [torch.empty((_electrons(k), 8), dtype=torch.float64, pin_memory=True) for k in members]
    if m["kind"] != "diag" and m["fields"]:
        state["grid"] = [torch.empty((9, *_ext(k)), dtype=torch.float64, pin_memory=True) for k in members]
    if m["kind"] in ("restore", "diag"):
        state["checkpoint"] = _checkpoint(m)
        state["sim"] = pic.Simulation(state["configs"][0], allocator=state["allocator"], stream=state["stream"])
        if m["kind"] == "diag":
            _restore(state["sim"], state.pop("checkpoint"), m)
    return state


def run(state):
    m = state["members"][0]
    if m["kind"] == "diag":
        sim = state["sim"]
        return {"energies": _own(torch.from_numpy(sim.energies()[:4]), m), "histogram": sim.histogram(96, 12.0, 36)}
    if m["kind"] == "restore":
        sim = state["sim"]
        _restore(sim, state["checkpoint"], m)
        sim.step(m["steps"])
        return _read(state, 0, sim)
    sims = [pic.Simulation(c, allocator=state["allocator"], stream=state["stream"]) for c in state["configs"]]
    if m["kind"] == "batch":
        pic.pic_batch_step([s.h for s in sims], m["steps"], state["stream"])
    else:
        sims[0].step(m["steps"])
    out = [_read(state, k, s) for k, s in enumerate(sims)]
    for s in sims:
        s.close()
    return out


_shared = {}


def _allocator():
    if "allocator" not in _shared:
        _shared["allocator"] = pic.torch_allocator()
    return _shared["allocator"]


def _ext(m):
    return tuple(m["n"][d] + 1 if d < m["dim"] else 1 for d in (2, 1, 0))


def _own(t, m):
    """Values in the precision that the simulation computed them in."""
    return t if m["precision"] == "fp64" else t.to(torch.float32)


def _restore(sim, chk, m):
    pic.pic_set_step(sim.h, m["focus_step"], sim.stream)
    sim.set_fields(chk["fields"])
    sim.set_particles(chk["x"], chk["u"], chk["w"], chk["id"])


def _read(state, k, sim):
    m = state["members"][k]
    out = {"energies": _own(torch.from_numpy(sim.energies()[:4]), m)}
    if m["fields"]:
        grid = state["grid"][k]
        pic.pic_diag(sim.h, pic.PIC_DIAG_FIELDS, grid.numpy(), sim.stream)
        out["fields"] = _own(grid.cuda(), m)
    if m["particles"]:
        host = state["records"][k]
        n = sim.info().n_alive
        pic.pic_diag(sim.h, pic.PIC_DIAG_PARTICLES, host[:n].numpy(), sim.stream)
        rec = host[:n].cuda()
        rows = torch.zeros((len(host), 7), dtype=torch.float64, device=rec.device)
        rows[rec[:, 7].long()] = rec[:, :7]
        out["x"], out["u"], out["w"] = (_own(v, m) for v in (rows[:, :m["dim"]], rows[:, 3:6], rows[:, 6]))
    return out


def _checkpoint(m):
    """A state as a running simulation has it: warm electrons spread over the slab, fields of a few
    per cent of the pulse.  Values that single precision holds, as a checkpoint of such a run has."""
    rng = np.random.default_rng([m["seed"], 11])
    n, dim = _electrons(m), m["dim"]
    off = rng.integers(0, 1 << 20, size=(n, 3), dtype=np.int64) / float(1 << 20)
    cell = _slab_cells(m)
    x = np.zeros((n, 3))
    x[:, :dim] = (cell + off[:, :dim]) * m["dx"]
    u = rng.standard_normal((n, 3), dtype=np.float32).astype(np.float64) * np.float32(0.4)
    u[:, 0] += 0.5
    u = u.astype(np.float32).astype(np.float64)
    w = np.full(n, np.float64(np.float32(m["n_e"] / m["ppc"])))
    fields = np.zeros((9, *_ext(m)))
    amp = 0.02 * m["a0"]
    grid = np.meshgrid(*[np.arange(e) for e in _ext(m)], indexing="ij")
    for comp in range(6):
        k = rng.uniform(0.02, 0.2, size=3)
        p = rng.uniform(0, TWO_PI, size=3)
        f = amp * np.cos(k[0] * grid[2] + p[0]) * np.cos(k[1] * grid[1] + p[1]) * np.cos(k[2] * grid[0] + p[2])
        sl = tuple(slice(0, m["n"][d] if _stag(comp, d) and d < dim else None) for d in (2, 1, 0))
        fields[comp][sl] = f[sl].astype(np.float32)
    return {"x": x, "u": u, "w": w, "id": np.arange(n, dtype=np.int64), "fields": fields}


# ---- what a pass cannot do without ----------------------------------------------------------
def work(case):
    """Per step: every electron's record read and written, per cell E and B read and written and J
    written and read once; the floating-point operations of gather, closed form, push and deposit.
    Beside the steps: a checkpoint restored, the state read back, a diagnostic's reads."""
    members = _members(case, 1)
    total = {"bytes": 0.0, "flops": 0.0}
    for m in members:
        es = 8 if m["precision"] == "fp64" else 4
        dim, ne, cells = m["dim"], _electrons(m), math.prod(e for e in _ext(m))
        gather = 2 * 6 * 3 ** dim
        closed = {"plane": 30, "gauss2d": 80, "lp": 280, "rp": 280}[m["beam"]]
        deposit = {1: 60, 2: 300, 3: 1100}[dim]
        if m["kind"] == "diag":
            total["bytes"] += ne * (4 * es + 4) + cells * 6 * es
            total["flops"] += cells * min(6, 2 ** dim) * closed
            continue
        record = 8 + (dim + 4) * es
        total["bytes"] += m["steps"] * (2 * ne * record + cells * es * 18)
        total["flops"] += m["steps"] * (ne * (gather + closed + 70 + deposit) + cells * 60)
        if m["kind"] == "restore":
            total["bytes"] += ne * 64 + cells * 9 * 8
        total["bytes"] += (ne * 64 if m["particles"] else 0) + (cells * 9 * 8 if m["fields"] else 0)
    return total


# ---- the same in 64 bits, plain torch -----------------------------------------------------
def exact(case, seed):
    c = _full(case)
    members = _members(case, seed)
    # seconds that it takes on this GPU, by measurement: a step's launches, its electrons, its grid
    cost = sum(m["steps"] * ({1: 0.0135, 2: 0.009, 3: 0.009}[m["dim"]] + _electrons(m) * {1: 0.0, 2: 2.5e-8, 3: 3.5e-8}[m["dim"]] +
                             math.prod(m["n"]) * (5e-8 if m["incident_grid"] else 4e-9)) for m in members)
    if cost > 21.0:
        return None
    if c["kind"] == "diag":
        r = _Reference(members[0], _checkpoint(members[0]))
        return {"energies": r.energies(), "histogram": r.histogram(96, 12.0, 36)}
    out = []
    for m in members:
        r = _Reference(m, _checkpoint(m) if c["kind"] == "restore" else None)
        for _ in range(m["steps"]):
            r.advance()
        o = {"energies": r.energies()}
        if m["fields"]:
            o["fields"] = r.F
        if m["particles"]:
            rows = torch.zeros((_electrons(m), 7), dtype=torch.float64, device=r.F.device)
            rows[r.id, : m["dim"]] = r.x.T
            rows[r.id, 3:6] = r.u.T
            rows[r.id, 6] = r.w
            o["x"], o["u"], o["w"] = rows[:, : m["dim"]], rows[:, 3:6], rows[:, 6]
        out.append(o)
    return out[0] if c["kind"] == "restore" else out


def _stag(comp, d):
    """Is component comp (Ex..Bz, Jx..Jz) half a cell up along axis d?"""
    return (d != comp % 3) if 3 <= comp < 6 else (d == comp % 3)


def _slab_cells(m):
    """Cells of the slab's electrons in the order of their ids: x fastest, ppc in each."""
    n = [m["hi"][d] - m["lo"][d] for d in range(m["dim"])]
    k = np.arange(_electrons(m), dtype=np.int64) // m["ppc"]
    out = np.empty((len(k), m["dim"]))
    for d in range(m["dim"]):
        out[:, d] = m["lo"][d] + k % n[d]
        k = k // n[d]
    return out


def _splitmix64(seed, k):
    """k-th outputs of SplitMix64 (Steele, Lea and Flood 2014)."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (k + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _pulse(m, X, Y, Z, tau):
    """Complex fields / (Psi0 / a^3) of the tightly focused pulse in its own frame (polarised along
    X or radially, propagating along Z): Psi = [g(tau + a(R + i)) - g(tau + a(-R + i))]/R with
    g = e^{i phi0} (1 - i tau/s)^-(s+1), R^2 = (X^2 + Y^2)/a^2 + (Z/a + i)^2."""
    a, s = m["a"], m["s"]
    xi, eta, zi = X / a, Y / a, Z / a + 1j
    u = xi * xi + eta * eta + zi * zi
    R = torch.sqrt(u)
    g = []
    for sign in (1.0, -1.0):
        w = 1.0 - 1j * (tau + a * (sign * R + 1j)) / s
        q = 1j * a / (s * w)
        g0 = np.exp(1j * m.get("phi0", 0.0)) * torch.exp(-(s + 1.0) * torch.log(w))
        g1 = (s + 1.0) * q * g0
        g.append((g0, g1, (s + 2.0) * q * g1))
    (p0, p1, p2), (m0, m1, m2) = g
    Pu = 0.5 * ((p1 + m1) / u - (p0 - m0) / (u * R))
    Puu = 0.25 * ((p2 - m2) / (u * R) - 3.0 * (p1 + m1) / (u * u) + 3.0 * (p0 - m0) / (u * u * R))
    PuD = 0.5 * ((p2 + m2) / u - (p1 - m1) / (u * R))
    PDD = (p2 - m2) / R
    if m["beam"] == "lp":
        lead = 2.0 * Pu - PDD + 2.0 * zi * PuD
        E = (lead + 4.0 * xi * xi * Puu, 4.0 * xi * eta * Puu, 4.0 * xi * zi * Puu - 2.0 * xi * PuD)
        B = (E[1], lead + 4.0 * eta * eta * Puu, 4.0 * eta * zi * Puu - 2.0 * eta * PuD)
    else:
        E = (4.0 * xi * zi * Puu, 4.0 * eta * zi * Puu, 2.0 * Pu + 4.0 * zi * zi * Puu - PDD)
        B = (2.0 * eta * PuD, -2.0 * xi * PuD, torch.zeros_like(E[0]))
    return E, B


def _focal_peak(m):
    """Largest on-axis field at the focus for Psi0 = 1 (E along X for lp, along Z for rp)."""
    tau = torch.linspace(-0.5, 0.5, 2001, dtype=torch.float64) * m["s"]
    zero = torch.zeros_like(tau)
    E, _ = _pulse({**m, "phi0": 0.0}, zero, zero, zero, tau)
    return float((E[0] if m["beam"] == "lp" else E[2]).abs().max()) / m["a"] ** 3


def _incident(m, x, t):
    """Incident E, B (six rows, grid axes) at the points x (one row per resolved axis), time t."""
    out = torch.zeros((6, x.shape[1]), dtype=torch.float64, device=x.device)
    if m["beam"] == "plane":
        xi = t - (x[0] - m["focus"][0])
        if m["gauss_envelope"]:
            c, env = m["t_focus"], torch.exp2(-4.0 * ((xi - m["t_focus"]) / m["duration"]) ** 2)
        else:
            c, T = m["duration"], m["duration"]
            env = torch.where((xi > 0) & (xi < 2 * T), torch.sin(math.pi * xi / (2 * T)) ** 2, torch.zeros_like(xi))
        out[1] = m["a0"] * torch.sin(xi - c + m["phi0"]) * env
        out[5] = out[1]
        return out
    Z = x[0] - m["focus"][0]
    X = x[1] - m["focus"][1]
    if m["beam"] == "gauss2d":
        zr = 0.5 * m["w0"] ** 2
        w2 = m["w0"] ** 2 * (1.0 + (Z / zr) ** 2)
        curv = Z / (Z * Z + zr * zr)
        env = torch.exp2(-4.0 * ((t - m["t_focus"] - Z) / m["duration"]) ** 2)
        amp = m["a0"] * (m["w0"] ** 2 / w2) ** 0.25 * torch.exp(-X * X / w2) * env
        ph = Z - t + 0.5 * X * X * curv - 0.5 * torch.atan(Z / zr) + m["phi0"]
        out[1] = amp * torch.cos(ph)
        out[5] = out[1]
        out[0] = amp * (2.0 * X / w2 * torch.sin(ph) - X * curv * torch.cos(ph))
        return out
    Y = x[2] - m["focus"][2] if m["dim"] > 2 else torch.zeros_like(Z)
    E, B = _pulse(m, X, Y, Z, t - m["t_focus"])
    k = m["psi0"] / m["a"] ** 3
    # the beam's z is the grid's x, its x the grid's y, its y the grid's z
    for row, f in enumerate((E[2], E[0], E[1], B[2], B[0], B[1])):
        out[row] = k * f.real
    return out


def _shape(d):
    """Order-2 weights of three neighbouring nodes, d the distance from the middle one."""
    return torch.stack([0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2])


class _Reference:
    """The scattered-field cycle in 64 bits; F[component][z][y][x], x[axis][electron]."""

    def __init__(self, m, chk):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.m, self.dev, self.dim = m, dev, m["dim"]
        self.step = m["focus_step"] if chk else 0
        self.F = torch.zeros((9, *_ext(m)), dtype=torch.float64, device=dev)
        self.left = 0.0
        n = _electrons(m)
        if chk:
            x, u, w = chk["x"][:, : self.dim], chk["u"], chk["w"]
            self.F[:] = torch.from_numpy(chk["fields"])
        else:
            p = np.arange(n, dtype=np.uint64)
            x = _slab_cells(m)
            for d in range(self.dim):
                x[:, d] += (_splitmix64(m["seed"], np.uint64(3) * p + np.uint64(d)) >> np.uint64(40)) / 16777216.0
            x *= m["dx"]
            u, w = np.zeros((n, 3)), np.full(n, m["n_e"] / m["ppc"])
            if m["supergauss"]:
                w *= 2.0 ** -(np.abs(2.0 * (x[:, 0] - m["prof"][0]) / m["prof"][1]) ** 12)
        self.x, self.u, self.w = (torch.from_numpy(np.ascontiguousarray(v.T)).to(dev) for v in (x, u, w))
        self.id = torch.arange(n, device=dev)

    def _nodes(self, comp):
        """Positions of all points of the grid for a component, one row per resolved axis."""
        m = self.m
        ax = [(torch.arange(m["n"][d] + 1, dtype=torch.float64, device=self.dev) + 0.5 * _stag(comp, d)) * m["dx"]
              if d < self.dim else torch.zeros(1, dtype=torch.float64, device=self.dev) for d in (2, 1, 0)]
        z, y, x = torch.meshgrid(*ax, indexing="ij")
        return torch.stack([v.reshape(-1) for v in (x, y, z)[: self.dim]])

    def _points(self, comp):
        """Slices of the points that a component has."""
        return tuple(slice(0, self.m["n"][d] + (0 if _stag(comp, d) else 1)) if d < self.dim else slice(0, 1)
                     for d in (2, 1, 0))

    def _total(self, t):
        """E, B of scattered plus incident field on the grid."""
        G = self.F[:6].clone()
        for comp in range(6):
            G[comp] += _incident(self.m, self._nodes(comp), t)[comp].reshape(G[comp].shape)
        return G

    def _gather(self, G, x):
        ez, ey, ex = _ext(self.m)
        stride = (1, ex, ex * ey)
        out = []
        for comp in range(6):
            idx, wt = torch.zeros((1, x.shape[1]), dtype=torch.int64, device=self.dev), 1.0
            for d in range(self.dim):
                y = x[d] / self.m["dx"] - 0.5 * _stag(comp, d)
                i = torch.floor(y + 0.5)
                w3 = _shape(y - i)
                i3 = (i.long() - 1 + torch.arange(3, device=self.dev)[:, None]) * stride[d]
                idx = (idx[None] + i3[:, None]).reshape(-1, x.shape[1])
                wt = w3 if d == 0 else (wt[None] * w3[:, None]).reshape(-1, x.shape[1])
            out.append((G[comp].reshape(-1)[idx] * wt).sum(0))
        return torch.stack(out)

    def _momentum(self, u, E, B):
        h = -0.5 * self.m["dt"]
        cross = lambda p, q: torch.linalg.cross(p, q, dim=0)  # noqa: E731
        if self.m["pusher"] == "boris":
            um = u + h * E
            t = h * B / torch.sqrt(1.0 + (um * um).sum(0))
            up = um + cross(um, t)
            return um + cross(up, 2.0 * t / (1.0 + (t * t).sum(0))) + h * E
        vay = self.m["pusher"] == "vay"
        if vay:
            w = u + h * (2.0 * E + cross(u / torch.sqrt(1.0 + (u * u).sum(0)), B))
        else:
            w = u + h * E
        tau = h * B                     # implicit midpoint rotation, gamma the positive root
        t2, ws = (tau * tau).sum(0), (w * tau).sum(0)
        sig, K = 1.0 + (w * w).sum(0) - t2, t2 + ws * ws
        t = tau / torch.sqrt(0.5 * (sig + torch.sqrt(sig * sig + 4.0 * K)))
        v = (w + (w * t).sum(0) * t + cross(w, t)) / (1.0 + (t * t).sum(0))
        return v if vay else 2.0 * v - w + h * E

    def _deposit(self, xo, xn, v, w):
        """Esirkepov's current of the straight moves xo -> xn (electron charge -1)."""
        m, N = self.m, xo.shape[1]
        ez, ey, ex = _ext(m)
        stride = (1, ex, ex * ey)
        S0, DS, base, off = [], [], 0, []
        for d in range(3):
            if d >= self.dim:
                S0.append(torch.ones((1, N), dtype=torch.float64, device=self.dev))
                DS.append(torch.zeros_like(S0[-1]))
                off.append(torch.zeros(1, dtype=torch.int64, device=self.dev))
                continue
            a, b = xo[d] / m["dx"], xn[d] / m["dx"]
            i0, i1 = torch.floor(a + 0.5), torch.floor(b + 0.5)
            s0 = torch.zeros((5, N), dtype=torch.float64, device=self.dev)
            s1 = torch.zeros_like(s0)
            s0[1:4] = _shape(a - i0)
            s1.scatter_(0, (i1 - i0).long() + torch.arange(1, 4, device=self.dev)[:, None], _shape(b - i1))
            S0.append(s0)
            DS.append(s1 - s0)
            base = base + (i0.long() - 2) * stride[d]
            off.append(torch.arange(5, device=self.dev) * stride[d])
        idx = base + (off[2][:, None, None] + off[1][None, :, None] + off[0][None, None, :])[..., None]
        view = {0: lambda q: q[None, None], 1: lambda q: q[None, :, None], 2: lambda q: q[:, None, None]}
        for c in range(3):
            p, q = [d for d in range(3) if d != c]
            Sp, Dp, Sq, Dq = view[p](S0[p]), view[p](DS[p]), view[q](S0[q]), view[q](DS[q])
            T = Sp * Sq + 0.5 * Dp * Sq + 0.5 * Sp * Dq + Dp * Dq / 3.0
            if c < self.dim:
                J = torch.cumsum(view[c](DS[c]) * T * (w * m["dx"] / m["dt"]), dim=2 - c)
            else:
                J = T * (-w * v[c])
            self.F[6 + c].reshape(-1).index_add_(0, idx.expand(J.shape).reshape(-1), J.reshape(-1))

    def advance(self):
        m, t = self.m, self.step * self.m["dt"]
        self.F[6:] = 0.0
        G = self._total(t) if m["incident_grid"] else self.F[:6]
        keep = torch.ones_like(self.w, dtype=torch.bool)
        for a in range(0, len(self.w), 1 << 18):
            p = slice(a, a + (1 << 18))
            x, w = self.x[:, p], self.w[p]
            EB = self._gather(G, x)
            if not m["incident_grid"]:
                EB = EB + _incident(m, x, t)
            u = self._momentum(self.u[:, p], EB[:3], EB[3:])
            v = u / torch.sqrt(1.0 + (u * u).sum(0))
            xn = x + m["dt"] * v[: self.dim]
            self._deposit(x, xn, v, w)
            self.x[:, p], self.u[:, p] = xn, u
            for d in range(self.dim):
                keep[p] &= (xn[d] >= 3 * m["dx"]) & (xn[d] < (m["n"][d] - 3) * m["dx"])
        if not bool(keep.all()):
            self.left += float(self._kinetic(self.u[:, ~keep], self.w[~keep]))
            self.x, self.u, self.w, self.id = self.x[:, keep], self.u[:, keep], self.w[keep], self.id[keep]
        self._yee()
        self.step += 1

    def _diff(self, A, d, sl):
        """Forward difference along axis d at the points sl."""
        if d >= self.dim:
            return 0.0
        up = list(sl)
        up[2 - d] = slice(sl[2 - d].start + 1, sl[2 - d].stop + 1)
        return (A[tuple(up)] - A[sl]) / self.m["dx"]

    def _faraday(self, h):
        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            sl = self._points(3 + c)
            self.F[3 + c][sl] -= h * (self._diff(self.F[b], a, sl) - self._diff(self.F[a], b, sl))

    def _yee(self):
        m, F = self.m, self.F
        old = F[:3].clone()
        self._faraday(0.5 * m["dt"])
        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            faces = [d for d in range(self.dim) if d != c]
            sl = list(self._points(c))
            for d in faces:
                sl[2 - d] = slice(1, m["n"][d])
            sl = tuple(sl)

            def back(A, d):
                lo = list(sl)
                if d >= self.dim:
                    return 0.0
                lo[2 - d] = slice(sl[2 - d].start - 1, sl[2 - d].stop - 1)
                return (A[sl] - A[tuple(lo)]) / m["dx"]

            F[c][sl] += m["dt"] * (back(F[3 + b], a) - back(F[3 + a], b) - F[6 + c][sl])
            # first-order Mur: faces, then (along the lower axis) the edges of two faces
            km = (m["dt"] - m["dx"]) / (m["dt"] + m["dx"])
            jobs = [({d: e}, d) for d in faces for e in (0, m["n"][d])]
            if len(faces) == 2:
                jobs += [({faces[0]: e, faces[1]: f}, faces[0]) for e in (0, m["n"][faces[0]]) for f in (0, m["n"][faces[1]])]
            for at, along in jobs:
                here, inward = list(sl), list(sl)
                for d, e in at.items():
                    here[2 - d] = inward[2 - d] = slice(e, e + 1)
                k = at[along] + (1 if at[along] == 0 else -1)
                inward[2 - along] = slice(k, k + 1)
                here, inward = tuple(here), tuple(inward)
                F[c][here] = old[c][inward] + km * (F[c][inward] - old[c][here])
        self._faraday(0.5 * m["dt"])

    def _kinetic(self, u, w):
        return (w * (torch.sqrt(1.0 + (u * u).sum(0)) - 1.0)).sum() * self.m["dx"] ** self.dim

    def energies(self):
        m, vol = self.m, self.m["dx"] ** self.dim
        G = self._total(self.step * m["dt"])
        es = sum(float((self.F[c][self._points(c)] ** 2).sum()) for c in range(6))
        et = sum(float((G[c][self._points(c)] ** 2).sum()) for c in range(6))
        return torch.tensor([0.5 * es * vol, 0.5 * et * vol, float(self._kinetic(self.u, self.w)), self.left],
                            dtype=torch.float64)

    def histogram(self, ne, emax, na):
        ek = torch.sqrt(1.0 + (self.u * self.u).sum(0)) - 1.0
        ang = torch.atan2(torch.sqrt(self.u[1] ** 2 + self.u[2] ** 2), self.u[0])
        ok = ek < emax
        k = (ek / emax * ne).long().clamp(0, ne - 1) * na + (ang / math.pi * na).long().clamp(0, na - 1)
        out = torch.zeros(ne * na, dtype=torch.float64, device=self.dev)
        return out.index_add_(0, k[ok], self.w[ok]).reshape(ne, na)
