"""Performance cases of the fluid-solute step, each through the entry points a user's program calls.

A case is one kind of run: a simulation advanced by a chunk of steps and read back into device
buffers, a step-by-step loop that reads the particle forces, a batch of ragged domains, or the
allocation-free binning of walkers. `run` advances the same simulation further each time it is
called. `exact` gives the fluid's outputs in binary64 with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_2308_05007_gb300 import inputs as I
from paper_2308_05007_gb300.rwmi import Batch, Simulation, bin_walkers_noalloc

DEV = "cuda"


def listed():
    return [
        # a dispersing plume of caller-owned walkers binned inside a pipeline that may not allocate
        {"name": "bin_100", "kind": "bin", "nx": 100, "ny": 100, "nz": 100, "walls": 0, "walkers": 1_000_000},
        # a host-side coupling loop: one step at a time, the force on every particle read after each
        {"name": "coupled_40x36x26", "kind": "coupled", "nx": 40, "ny": 36, "nz": 26, "walls": 4, "q": 19,
         "storage": 1, "particles": 3, "walkers": 3000, "steps": 8},
        # the smallest request of the served stream: latency and launches
        {"name": "request_33", "kind": "request", "n": 33, "q": 15, "storage": 1, "particles": 1,
         "walkers": 70_000, "steps": 32},
        # Section 3.1's point source at the paper's size: walkers only in a uniform stream
        {"name": "point_source_100", "kind": "point", "n": 100, "q": 19, "walkers": 1_000_000, "steps": 32},
        # a middling request of the served stream with binary16 populations
        {"name": "request_fp16_117", "kind": "request", "n": 117, "q": 15, "storage": 2, "particles": 3,
         "walkers": 1_000_000, "steps": 32},
        # many small ragged domains advanced together
        {"name": "batch_64", "kind": "batch", "domains": 64, "edge_lo": 16, "edge_hi": 48, "steps": 64},
        # the paper's oscillator box (50 particles, 2e6 walkers) with its own coupling: free
        # particles, interpolated bounce-back, D3Q19
        {"name": "paper_dem_ibb", "kind": "dem", "nx": 120, "ny": 120, "nz": 180, "q": 19, "storage": 1,
         "coupling": 1, "particles": 50, "walkers": 2_000_000, "steps": 16},
        # the binary64 run that separates the method's error from rounding, at the oracle's size
        {"name": "precision_96_fp64", "kind": "precision", "n": 96, "storage": 3, "particles": 4,
         "walkers": 20_000, "steps": 16},
        # the oscillator workload: moving particles, no-slip walls, 1e7 walkers
        {"name": "oscillator_256", "kind": "oscillator", "n": 256, "q": 15, "storage": 1, "coupling": 0,
         "particles": 64, "walkers": 10_000_000, "steps": 32},
        # the same with the paper's velocity set and binary16 populations
        {"name": "oscillator_256_q19_fp16", "kind": "oscillator", "n": 256, "q": 19, "storage": 2, "coupling": 0,
         "particles": 64, "walkers": 10_000_000, "steps": 16},
        # the same with the paper's interpolated bounce-back
        {"name": "oscillator_256_ibb", "kind": "oscillator", "n": 256, "q": 15, "storage": 1, "coupling": 1,
         "particles": 64, "walkers": 10_000_000, "steps": 16},
        # the precision workload: static particles, 3e7 walkers; the largest
        {"name": "precision_384", "kind": "precision", "n": 384, "storage": 1, "particles": 128,
         "walkers": 30_000_000, "steps": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bin", "coupled", "request", "request", "point", "batch", "dem", "precision", "oscillator",
                       "oscillator"])
    if kind == "bin":
        return {"kind": kind, "nx": rng.randint(16, 101), "ny": rng.randint(16, 101), "nz": rng.randint(16, 101),
                "walls": rng.choice([0, 4]), "walkers": _log(rng, 10_000, 1_000_000)}
    if kind == "coupled":
        return {"kind": kind, "nx": rng.randint(36, 72), "ny": rng.randint(34, 72), "nz": rng.randint(26, 72),
                "walls": rng.choice([0, 4]), "q": rng.choice([15, 19]), "storage": rng.choice([0, 1]), "particles": 3,
                "walkers": _log(rng, 3000, 100_000), "steps": 8}
    if kind == "request":
        n = _log(rng, 32, 240)
        return {"kind": kind, "n": n, "q": 15, "storage": rng.choice([1, 2]), "particles": rng.randint(1, 4),
                "walkers": min(2 * n ** 3, _log(rng, 100_000, 10_000_000)), "steps": 16 * rng.randint(1, 2)}
    if kind == "point":
        return {"kind": kind, "n": rng.randint(50, 120), "q": rng.choice([15, 19]),
                "walkers": _log(rng, 100_000, 3_000_000), "steps": 16 * rng.randint(1, 3)}
    if kind == "batch":
        if rng.random() < 0.5:
            return {"kind": kind, "domains": rng.randint(24, 128), "edge_lo": 16, "edge_hi": 48, "steps": 64}
        return {"kind": kind, "domains": rng.randint(8, 24), "edge_lo": 48, "edge_hi": 160, "steps": 32}
    if kind == "dem":
        return {"kind": kind, "nx": rng.randint(80, 140), "ny": rng.randint(80, 140), "nz": rng.randint(90, 190),
                "q": rng.choice([15, 19]), "storage": 1, "coupling": rng.choice([0, 1]),
                "particles": rng.randint(10, 60), "walkers": _log(rng, 100_000, 3_000_000), "steps": 16}
    if kind == "precision":
        storage = rng.choice([0, 1, 2, 3])
        n = _log(rng, 64, 110) if storage == 3 else _log(rng, 96, 340)
        return {"kind": kind, "n": n, "storage": storage, "particles": max(1, int(128 * (n / 384.0) ** 3)),
                "walkers": int(30_000_000 * (n / 384.0) ** 3), "steps": 16}
    n = rng.randint(128, 272)
    return {"kind": kind, "n": n, "q": rng.choice([15, 19]), "storage": 1, "coupling": rng.choice([0, 1]),
            "particles": max(2, int(64 * (n / 256.0) ** 3)), "walkers": int(10_000_000 * (n / 256.0) ** 3), "steps": 16}


# ------------------------------------------------------------------------------------------
# Inputs: the seeded workloads of the repository
# ------------------------------------------------------------------------------------------
def _placed(place, n_particles):
    """place(P) with one particle fewer each time the box is too crowded."""
    while True:
        try:
            return place(n_particles)
        except RuntimeError:
            if n_particles <= 1:
                raise
            n_particles -= 1


def _workload(case, seed):
    kind = case["kind"]
    if kind == "coupled":
        return _placed(lambda p: I.ragged(dims=(case["nx"], case["ny"], case["nz"]), n_particles=p,
                                          n_walkers=case["walkers"], seed=seed, walls=case["walls"], q=case["q"],
                                          storage=case["storage"]), case["particles"])
    if kind == "point":
        w = I.point_source(n=case["n"], n_walkers=case["walkers"], velocity=(0.2, 0.0, 0.0), seed=seed)
        return I.with_(w, q=case["q"])
    if kind == "precision":
        return _placed(lambda p: I.precision(n=case["n"], n_particles=p, n_walkers=case["walkers"], seed=seed,
                                             storage=case["storage"]), case["particles"])
    if kind == "oscillator":
        w = _placed(lambda p: I.oscillator(n=case["n"], n_particles=p, n_walkers=case["walkers"], morph_seed=seed,
                                           seed=seed, q=case["q"], storage=case["storage"]), case["particles"])
        return I.with_(w, coupling=case["coupling"])
    if kind == "dem":
        w = _placed(lambda p: I.dem_box(dims=(case["nx"], case["ny"], case["nz"]), n_particles=p, seed=seed,
                                        n_walkers=case["walkers"], storage=case["storage"], q=case["q"]),
                    case["particles"])
        return I.with_(w, coupling=case["coupling"])
    # a request of the served stream: resting clusters of 1-6 centres in a periodic box
    n, rng = case["n"], np.random.default_rng(seed)
    ks = min(1.0, (n / 64.0) ** 2)
    mb = _placed(lambda p: I.random_metaballs(rng, p, (n, n, n), 0, n_centers=(1, 6), sigma=3.0 * math.sqrt(ks),
                                              k_range=(20.0 * ks, 60.0 * ks), max_tries=2000), case["particles"])
    return I.Workload(name="request", dims=(n, n, n), tau=float(rng.uniform(0.6, 1.0)),
                      D=float(rng.uniform(0.001, 0.02)), seed=seed, q=case["q"], body_force=(1e-6, 0.0, 0.0),
                      metaballs=mb, n_walkers=case["walkers"], walker_box=((0.0,) * 3, (float(n),) * 3),
                      storage=case["storage"])


def _workloads(case, seed):
    if case["kind"] != "batch":
        return [_workload(case, seed)]
    big = case["edge_hi"] > 64
    ws = I.batched(n_domains=case["domains"], edge=(case["edge_lo"], case["edge_hi"]),   # the domains' sizes and shapes
                   particles=(4, 32) if big else (1, 4), centers=(2, 10) if big else (2, 4),
                   walkers=(100_000, 2_000_000) if big else (2000, 40_000))
    rng = np.random.default_rng(seed)
    for k, w in enumerate(ws):   # walkers, drive phase, viscosity and diffusion of this seed
        w.seed, w.tau, w.D = seed * 1000 + k, float(rng.uniform(0.6, 1.0)), float(rng.uniform(0.001, 0.02))
        w.metaballs.phase[:] = rng.uniform(0.0, 2.0 * math.pi)
    return ws


def _plume(case, seed):
    """Walkers of a dispersing plume in random order: (x, y, z, mass), unwrapped."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    dims = torch.tensor([case["nx"], case["ny"], case["nz"]], device=DEV, dtype=torch.float32)
    pos = torch.ones((case["walkers"], 4), device=DEV, dtype=torch.float32)
    pos[:, :3] = dims * (0.5 + 0.15 * torch.randn((case["walkers"], 3), generator=gen, device=DEV))
    pos[:, 0] += 3.0 * dims[0]   # drifted downstream through a few periods
    return pos


def prepare(case, seed):
    if case["kind"] == "bin":
        pos = _plume(case, seed)
        return {"case": case, "pos": pos, "sorted": torch.empty_like(pos),
                "counts": torch.empty(case["nx"] * case["ny"] * case["nz"], dtype=torch.int32, device=DEV)}
    ws = _workloads(case, seed)
    sims = [Simulation.from_workload(w, sort_interval=16) for w in ws]
    cells = sum(s.n_cells for s in sims)
    state = {"case": case, "sims": sims, "batch": Batch(sims) if case["kind"] == "batch" else None,
             "u": torch.empty((cells, 3), dtype=torch.float32, device=DEV),
             "rho": torch.empty(cells, dtype=torch.float32, device=DEV),
             "conc": torch.empty(cells, dtype=torch.int32, device=DEV),
             "mom": torch.empty((len(sims), 13), dtype=torch.float64, device=DEV)}
    if case.get("storage") == 3:   # the error study reads the populations themselves
        state["f"] = torch.empty((sims[0].q, cells), dtype=torch.float64, device=DEV)
    return state


# ------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "bin":
        bin_walkers_noalloc((case["nx"], case["ny"], case["nz"]), case["walls"], state["pos"], state["counts"],
                            state["sorted"], stream=torch.cuda.current_stream())
        return {"counts": state["counts"], "sorted": state["sorted"]}
    sims, out = state["sims"], {}
    if case["kind"] == "coupled":
        forces = []
        for _ in range(case["steps"]):
            sims[0].step(1)
            forces.append(sims[0].particle_forces())
        # summed from binary32 populations: kept as binary32
        out["forces"] = np.asarray(forces, np.float32)
    elif state["batch"] is not None:
        state["batch"].step(case["steps"])
        state["batch"].sync()
    else:
        sims[0].step(case["steps"])
    at = 0
    for k, s in enumerate(sims):
        end = at + s.n_cells
        s.velocity(out=state["u"][at:end])
        s.density(out=state["rho"][at:end])
        s.concentration(out=state["conc"][at:end])
        s.walker_moments(out=state["mom"][k])
        at = end
    out.update(velocity=state["u"], density=state["rho"], concentration=state["conc"], moments=state["mom"])
    if "f" in state:
        out["populations"] = sims[0].populations(out=state["f"])
    if case["kind"] == "dem":
        out["particles"] = sims[0].particle_state()
    return out


def work(case):
    """Bytes: per cell and step the populations read and written and the velocity written and read,
    per walker and step its position read and written, and the outputs. Operations: the moments,
    equilibrium, relaxation and forcing per direction, the interpolation and noise per walker."""
    if case["kind"] == "bin":
        return {"bytes": 32.0 * case["walkers"] + 4.0 * case["nx"] * case["ny"] * case["nz"],
                "flops": 12.0 * case["walkers"]}
    if case["kind"] == "batch":
        ws = _workloads(case, 1)
        cells, walkers, q = sum(w.n_cells for w in ws), sum(w.n_walkers for w in ws), 15
    else:
        n = case.get("n", 0)
        cells = n ** 3 if n else case["nx"] * case["ny"] * case["nz"]
        walkers, q = case["walkers"], case.get("q", 15)
    s = {0: 4, 1: 4, 2: 2, 3: 8}[case.get("storage", 1)]
    out = 20.0 * cells + (8.0 * q * cells if s == 8 else 0.0)
    return {"bytes": case["steps"] * (cells * (2.0 * q * s + 24.0) + 32.0 * walkers) + out,
            "flops": case["steps"] * (cells * (14.0 * q + 20.0) + 120.0 * walkers)}


# ------------------------------------------------------------------------------------------
# The fluid in binary64: BGK with Guo forcing on partially saturated cells (prescribed particles),
# half-way bounce-back at walls, pull streaming, in plain torch operations
# ------------------------------------------------------------------------------------------
HALF = {15: [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1), (1, 1, -1), (1, -1, 1), (1, -1, -1)],
        19: [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]}
WEIGHT = {15: {0: 2 / 9, 1: 1 / 9, 3: 1 / 72}, 19: {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}}


def _pose(w, p, t):
    """Origin, velocity and rotation of particle p at step t."""
    mb = w.metaballs
    s = c = 0.0
    if mb.period[p] > 0:
        th = 2 * math.pi * t / mb.period[p] + mb.phase[p]
        s, c = math.sin(th), math.cos(th) * 2 * math.pi / mb.period[p]
    spin = mb.omega[p]
    R, wn = np.eye(3), float(np.linalg.norm(spin))
    if wn > 0:
        a = spin / wn
        K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
        R = math.cos(wn * t) * np.eye(3) + math.sin(wn * t) * K + (1 - math.cos(wn * t)) * np.outer(a, a)
    return mb.origin[p] + mb.amplitude[p] * s, mb.amplitude[p] * c, R, spin


def _minimum(d, n, wall):
    return d if wall else torch.where(d > 0.5 * n, d - n, torch.where(d < -0.5 * n, d + n, d))


def _solid(w, t, cnt, us):
    """Adds every particle's sub-sample count (binary32 inside test, Eq. 3) and rigid velocity at
    its cells at step t; the particles keep apart, so no cell has sub-samples of two of them
    unless they share it, where the larger share owns it."""
    mb, dims = w.metaballs, w.dims
    wall = [bool(w.wall_mask >> a & 1) for a in range(3)]
    cnt.zero_()
    most = torch.zeros_like(cnt)
    for p in range(mb.n_particles):
        sl = slice(int(mb.center_offsets[p]), int(mb.center_offsets[p + 1]))
        body = mb.centers_body[sl].astype(np.float64)
        k = mb.k[sl]
        org, vel, R, spin = _pose(w, p, t)
        centre = org + body @ R.T
        reach = float(np.linalg.norm(body, axis=1).max() + math.sqrt(k.astype(np.float64).sum())) + 1.0
        idx = []
        for a in range(3):
            lo, hi = int(math.floor(org[a] - reach)), int(math.ceil(org[a] + reach))
            if wall[a]:
                i = np.arange(max(lo, 0), min(hi, dims[a]))
            else:
                centre[:, a] -= dims[a] * np.floor(centre[:, a] / dims[a])
                i = np.arange(lo, hi) % dims[a] if hi - lo < dims[a] else np.arange(dims[a])
            idx.append(torch.from_numpy(i.astype(np.int64)).to(DEV))
        sub = torch.tensor([0.125, 0.375, 0.625, 0.875], device=DEV)
        x, y, z = [(i.to(torch.float32)[:, None] + sub).reshape(-1) for i in idx]
        f = None
        for m, c in enumerate(centre.astype(np.float32)):
            dx, dy, dz = [_minimum(v - float(c[a]), float(dims[a]), wall[a]) for a, v in enumerate((x, y, z))]
            xy = (dx * dx)[None, :] + (dy * dy)[:, None]
            term = torch.full((), float(k[m]), dtype=torch.float32, device=DEV) / (xy[None] + (dz * dz)[:, None, None])
            f = term if f is None else f + term
        inside = (f >= 1.0).to(torch.int32)
        shape = (len(idx[2]), 4, len(idx[1]), 4, len(idx[0]), 4)
        n = inside.reshape(shape).sum((1, 3, 5)).to(cnt.dtype)
        at = (idx[2][:, None, None], idx[1][None, :, None], idx[0][None, None, :])
        cnt[at] += n
        own = n > most[at]
        most[at] = torch.maximum(most[at], n)
        if not (np.any(vel) or np.any(spin)):
            continue
        r = [_minimum(i.to(torch.float64) + 0.5 - (org[a] if wall[a] else org[a] % dims[a]), float(dims[a]), wall[a])
             for a, i in enumerate(idx)]
        rx, ry, rz = r[0][None, None, :], r[1][None, :, None], r[2][:, None, None]
        v = (vel[0] + spin[1] * rz - spin[2] * ry, vel[1] + spin[2] * rx - spin[0] * rz,
             vel[2] + spin[0] * ry - spin[1] * rx)
        for a in range(3):
            us[a][at] = torch.where(own, v[a].expand(n.shape), us[a][at])


def _fluid(w, steps):
    """(velocity, density, populations) after `steps` steps from rest (or the initial velocity)."""
    q, (nx, ny, nz), tau = w.q, w.dims, w.tau
    e = [(0, 0, 0)] + HALF[q] + [tuple(-c for c in d) for d in HALF[q]]
    H = len(HALF[q])
    opp = [0] + list(range(H + 1, 2 * H + 1)) + list(range(1, H + 1))
    wt = [WEIGHT[q][sum(c * c for c in d)] for d in e]
    wall = [bool(w.wall_mask >> a & 1) for a in range(3)]
    shape = (nz, ny, nx)
    new = lambda: torch.zeros(shape, dtype=torch.float64, device=DEV)  # noqa: E731
    u0 = w.init_velocity
    uu0 = sum(c * c for c in u0)
    f = []
    for d, wi in zip(e, wt):
        eu = sum(a * b for a, b in zip(d, u0))
        f.append(new() + wi * w.rho0 * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * uu0))
    P = w.metaballs.n_particles if w.metaballs is not None else 0
    moving = P and (np.any(w.metaballs.amplitude) or np.any(w.metaballs.omega))
    cnt, us, B = new(), [new(), new(), new()], None
    for t in range(steps):
        if P and (t == 0 or moving):
            for v in us:
                v.zero_()
            _solid(w, t, cnt, us)
            eps = cnt / 64.0
            B = eps * (tau - 0.5) / ((1.0 - eps) + (tau - 0.5))
        s = math.sin(2 * math.pi * t / w.force_period) if w.force_period > 0 else 1.0
        F = [c * s for c in w.body_force]
        g = []
        for i, d in enumerate(e):   # pull
            v = torch.roll(f[i], (d[2], d[1], d[0]), (0, 1, 2)) if any(d) else f[i].clone()
            for a, ax in ((0, 2), (1, 1), (2, 0)):
                if wall[a] and d[a]:
                    at = 0 if d[a] > 0 else w.dims[a] - 1
                    v.select(ax, at).copy_(f[opp[i]].select(ax, at))
            g.append(v)
        f = None
        rho = sum(g)
        j = [new() + 0.5 * F[a] for a in range(3)]
        for i, d in enumerate(e):
            for a in range(3):
                if d[a]:
                    j[a] += d[a] * g[i]
        u = [c / rho for c in j]
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        ss = us[0] * us[0] + us[1] * us[1] + us[2] * us[2] if P else None

        def dot(d, v):
            out = 0.0
            for a in range(3):
                if d[a]:
                    out = out + d[a] * v[a]
            return out

        f = []
        for i, d in enumerate(e):
            eu, eF = dot(d, u), dot(d, F)
            fe = wt[i] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * uu)
            S = (1 - 0.5 / tau) * wt[i] * (3 * (eF - uF) + 9 * eu * eF)
            relax = S - (g[i] - fe) / tau
            if P:
                es, eo = dot(d, us), -1.0 * eu
                solid = (g[opp[i]] - wt[i] * rho * (1 + 3 * eo + 4.5 * eu * eu - 1.5 * uu) - g[i]
                         + wt[i] * rho * (1 + 3 * es + 4.5 * es * es - 1.5 * ss))
                relax = (1 - B) * relax + B * solid
            f.append(g[i] + relax)
        del g
    return torch.stack(u, -1).reshape(-1, 3), sum(f).reshape(-1), f


def exact(case, seed):
    if case["kind"] in ("bin", "dem") or case.get("coupling"):
        return None
    if case.get("domains", 1) * case["steps"] > 4096:
        return None   # thousands of small launches per step of every domain: too long
    parts = [_fluid(w, case["steps"]) for w in _workloads(case, seed)]
    out = {"velocity": torch.cat([p[0] for p in parts]), "density": torch.cat([p[1] for p in parts]),
           "concentration": None, "moments": None}
    if case["kind"] == "coupled":
        out["forces"] = None
    if case.get("storage") == 3:
        out["populations"] = torch.stack([v.reshape(-1) for v in parts[0][2]])
    return out
