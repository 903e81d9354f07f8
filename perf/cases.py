"""The solver's performance cases: what users of the package run, over the
range of sizes, lattices, storages and options it serves.

Every case goes through the public entry points (lbm.Lattice, lbm.Batch,
serve.Server) and returns whole fields.  ``listed()`` names the cases,
``draw()`` gives further ones of the same ranges, ``prepare()`` builds what a
user's program holds before the call (inputs made from the seed, lattice
handles, a batch, a server), ``run()`` is one pass, ``work()`` its
unavoidable traffic and arithmetic, and ``exact()`` the same pass in 64 bits
by a plain torch restatement of the scheme.

Kinds of case:

* ``solve``      -- one short solve from rest on a static volume fraction:
                    initialise, step, read rho, p, u and the check sums.
* ``transient``  -- phi and a force field given anew before every step, as the
                    manufactured-solution validation runs do (FP64 mostly).
* ``wave``       -- a travelling-wave volume fraction evaluated on the device
                    and refreshed every 10 steps (the benchmark's workload).
* ``staged``     -- phi snapshots in pinned host memory, staged to the device
                    while the previous steps run.
* ``porous``     -- a channel through smoothed random spheres with walls on y,
                    optionally with the drag law and the Smagorinsky closure.
* ``batch``      -- many independent lattices advanced together.
* ``serve``      -- a burst of host requests through the request server.
"""
from __future__ import annotations

import itertools
import math
import random

import numpy as np
import torch

from paper_2208_09267_gb300 import inputs, lbm, serve

DEV = "cuda"
STEPS_PER_REFRESH = 10
WAVE_PERIOD = 1000.0     # steps per period of the travelling wave
G = 1e-6                 # body force of the workloads, along x
ELEM = {"fp64": 8, "fp32": 4, "fp16": 2}
Q_OF = {"D1Q3": 3, "D2Q9": 9, "D3Q19": 19, "D3Q27": 27}


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest work: the 2D validation case in FP64, 1000 steps from
        # rest on 64 x 64 cells; latency of dependent steps
        {"name": "d2q9_64_fp64_solve", "kind": "solve", "lattice": "D2Q9", "nx": 64, "ny": 64, "nz": 1,
         "storage": "fp64", "tau": 0.8, "walls": 0, "steps": 1000},
        # order-of-convergence runs: D3Q27 in FP64, phi and the manufactured
        # force of every step handed over on the device before it
        {"name": "d3q27_48_fp64_transient", "kind": "transient", "lattice": "D3Q27", "nx": 48, "ny": 48, "nz": 48,
         "storage": "fp64", "tau": 0.53, "steps": 40},
        # one small 3D solve of odd sides, the step budget of a short request
        {"name": "d3q19_61x75x67_fp32_solve", "kind": "solve", "lattice": "D3Q19", "nx": 61, "ny": 75, "nz": 67,
         "storage": "fp32", "tau": 0.6, "walls": 0, "steps": 500},
        # a coupled run: snapshots of phi arrive from the host every 10 steps
        {"name": "d3q19_128_fp16_staged", "kind": "staged", "lattice": "D3Q19", "nx": 128, "ny": 128, "nz": 128,
         "storage": "fp16", "tau": 0.6, "steps": 100},
        # the benchmark's headline workload in both storages
        {"name": "d3q19_256_fp32_wave", "kind": "wave", "lattice": "D3Q19", "nx": 256, "ny": 256, "nz": 256,
         "storage": "fp32", "tau": 0.6, "steps": 100},
        {"name": "d3q19_256_fp16_wave", "kind": "wave", "lattice": "D3Q19", "nx": 256, "ny": 256, "nz": 256,
         "storage": "fp16", "tau": 0.6, "steps": 100},
        # the largest: the porous channel of the benchmark in both storages
        {"name": "d3q27_512_fp32_porous", "kind": "porous", "lattice": "D3Q27", "nx": 512, "ny": 256, "nz": 256,
         "storage": "fp32", "tau": 0.6, "steps": 50, "drag": False, "les": 0.0},
        {"name": "d3q27_512_fp16_porous", "kind": "porous", "lattice": "D3Q27", "nx": 512, "ny": 256, "nz": 256,
         "storage": "fp16", "tau": 0.6, "steps": 50, "drag": False, "les": 0.0},
        # a packed bed with the drag law and the Smagorinsky closure
        {"name": "d3q19_150x96x90_fp32_drag", "kind": "porous", "lattice": "D3Q19", "nx": 150, "ny": 96, "nz": 90,
         "storage": "fp32", "tau": 0.55, "steps": 50, "drag": True, "les": 0.1},
        # independent lattices of mixed size, half 2D and half 3D, in FP16
        {"name": "batch_32_mixed_fp16", "kind": "batch", "storage": "fp16", "squares": 16, "cubes": 16,
         "square_min": 32, "square_max": 512, "cube_min": 32, "cube_max": 128, "sizes_seed": 11, "steps": 50},
        # many small 2D lattices in FP32: a parameter sweep
        {"name": "batch_64_small_fp32", "kind": "batch", "storage": "fp32", "squares": 64, "cubes": 0,
         "square_min": 32, "square_max": 96, "cube_min": 32, "cube_max": 32, "sizes_seed": 12, "steps": 100},
        # a burst of requests from the host, results back on the host
        {"name": "serve_6_fp16", "kind": "serve", "storage": "fp16", "requests": 6, "side_min": 32, "side_max": 96,
         "step_min": 150, "step_max": 400, "sizes_seed": 13},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "transient", "wave", "staged", "porous", "porous", "batch", "serve"])
    low = rng.choice(["fp32", "fp16"])
    if kind == "solve":
        lattice = rng.choice(["D2Q9", "D2Q9", "D3Q19", "D3Q19", "D3Q27", "D1Q3"])
        storage = rng.choice(["fp64", "fp32", "fp32", "fp16"])
        walls = rng.choice([0, 0, 2])
        if lattice == "D1Q3":
            shape, walls = (_log_int(rng, 32, 4096), 1, 1), 0
        elif lattice == "D2Q9":
            hi = 256 if storage == "fp64" else 640
            shape = (_log_int(rng, 16, hi), _log_int(rng, 16, hi), 1)
        else:
            hi = 40 if storage == "fp64" else 160
            shape = tuple(_log_int(rng, 16, hi) for _ in range(3))
        return {"kind": kind, "lattice": lattice, "nx": shape[0], "ny": shape[1], "nz": shape[2], "storage": storage,
                "tau": round(rng.uniform(0.55, 1.2), 3), "walls": walls, "steps": _log_int(rng, 60, 500)}
    if kind == "transient":
        storage = rng.choice(["fp64", "fp64", "fp32"])
        lattice = rng.choice(["D2Q9", "D3Q27"])
        n = _log_int(rng, 32, 128) if lattice == "D2Q9" else _log_int(rng, 16, 48)
        return {"kind": kind, "lattice": lattice, "nx": n, "ny": n, "nz": 1 if lattice == "D2Q9" else n,
                "storage": storage, "tau": round(rng.uniform(0.53, 0.7), 3), "steps": rng.randint(10, 40)}
    if kind in ("wave", "staged"):
        top = 256 if kind == "wave" else 160
        shape = [_log_int(rng, 48, top) for _ in range(3)]
        return {"kind": kind, "lattice": "D3Q19", "nx": shape[0], "ny": shape[1], "nz": shape[2], "storage": low,
                "tau": round(rng.uniform(0.55, 0.8), 3), "steps": 10 * rng.randint(3, 10)}
    if kind == "porous":
        special = rng.random() < 0.4
        top = 192 if special else 512
        return {"kind": kind, "lattice": rng.choice(["D2Q9", "D3Q19", "D3Q27"]), "nx": _log_int(rng, 48, top),
                "ny": _log_int(rng, 32, 192), "nz": _log_int(rng, 32, 160), "storage": low,
                "tau": round(rng.uniform(0.55, 0.8), 3), "steps": rng.randint(20, 50), "drag": special,
                "les": rng.choice([0.0, 0.1]) if special else 0.0}
    if kind == "batch":
        top = rng.choice([96, 256, 512])
        return {"kind": kind, "storage": low, "squares": rng.randint(2, 16), "cubes": rng.randint(0, 12),
                "square_min": 32, "square_max": top, "cube_min": 32, "cube_max": max(32, top // 4),
                "sizes_seed": rng.randint(1, 10 ** 6), "steps": 2 * rng.randint(10, 50)}
    return {"kind": "serve", "storage": low, "requests": rng.randint(2, 6), "side_min": 32,
            "side_max": rng.choice([48, 64, 96]), "step_min": 100, "step_max": 400,
            "sizes_seed": rng.randint(1, 10 ** 6)}


# --------------------------------------------------- sizes that a case fixes

def _shape(case):
    """(nx, ny, nz) of a single-lattice case."""
    return case["nx"], case["ny"], 1 if case["lattice"] in ("D2Q9", "D1Q3") else case["nz"]


def _members(case):
    """(lattice, side) of every member of a batch."""
    r = random.Random(case["sizes_seed"])
    out = [("D2Q9", r.randint(case["square_min"], case["square_max"])) for _ in range(case["squares"])]
    return out + [("D3Q19", r.randint(case["cube_min"], case["cube_max"])) for _ in range(case["cubes"])]


def _requests(case):
    """(side, steps) of every request of a burst."""
    r = random.Random(case["sizes_seed"])
    return [(_log_int(r, case["side_min"], case["side_max"]), _log_int(r, case["step_min"], case["step_max"]))
            for _ in range(case["requests"])]


def _walls(case):
    return 2 if case["kind"] == "porous" else case.get("walls", 0)


# ------------------------------------------------------------------- inputs

def _gen(seed, salt=0):
    return np.random.default_rng([20220819, int(seed), salt])


def _sine(lattice, shape, amp, phases, dtype, device=DEV):
    """(1 - amp) + amp prod_a sin(2 pi x_a / n_a + phase_a), shape (nz, ny, nx)."""
    nx, ny, nz = shape
    ax = [torch.sin(2 * math.pi * torch.arange(n, dtype=torch.float64, device=device) / n + ph)
          for n, ph in zip((nx, ny, nz), phases)]
    s = ax[0].reshape(1, 1, nx)
    if lattice != "D1Q3":
        s = s * ax[1].reshape(1, ny, 1)
    if lattice in ("D3Q19", "D3Q27"):
        s = s * ax[2].reshape(nz, 1, 1)
    return ((1.0 - amp) + amp * s).to(dtype).contiguous()


def _close_walls(phi):
    """Wall layers on y carry the phi of their fluid neighbour."""
    phi[:, 0] = phi[:, 1]
    phi[:, -1] = phi[:, -2]
    return phi


def _spheres(shape, seed, packing=0.35, rmin=4.0, rmax=12.0, sigma=3.0, phi_min=0.4):
    """phi = 1 - (1 - phi_min) (Gaussian * indicator of random spheres) with
    walls on y, float32 on the device; disks where nz = 1."""
    nx, ny, nz = shape
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 7919 + 1)
    flat = nz == 1
    p = 3 if flat else 4     # moments of U[rmin, rmax]
    mean = (rmax ** p - rmin ** p) / (p * (rmax - rmin))
    vol = math.pi * mean if flat else 4.0 / 3.0 * math.pi * mean
    count = max(1, int(math.ceil(-math.log(1.0 - packing) * nx * ny * nz / vol)))
    centre = torch.rand(count, 3, generator=gen, device=DEV)
    radius = rmin + (rmax - rmin) * torch.rand(count, generator=gen, device=DEV)
    ext = torch.tensor([nx, ny, nz], device=DEV)
    centre = centre * ext
    if flat:
        centre[:, 2] = 0.0
    w = int(rmax) + 1
    r = torch.arange(-w, w + 1, device=DEV)
    off = torch.cartesian_prod(r[:1] * 0 if flat else r, r, r).flip(1)     # (x, y, z) offsets
    chi = torch.zeros(nx * ny * nz, dtype=torch.float32, device=DEV)
    for a in range(0, count, 512):
        base = torch.floor(centre[a:a + 512]).long()[:, None, :] + off[None]
        inside = (base - centre[a:a + 512, None, :]).square().sum(2) <= radius[a:a + 512, None].square()
        inside &= (base[..., 1] >= 0) & (base[..., 1] < ny)
        cell = base[inside] % ext
        chi[(cell[:, 2] * ny + cell[:, 1]) * nx + cell[:, 0]] = 1.0
    chi = chi.reshape(nz, ny, nx)
    k = np.exp(-0.5 * (np.arange(-9, 10) / sigma) ** 2)
    k /= k.sum()
    for dim, n in ((2, nx), (1, ny), (0, nz)):
        if n == 1:
            continue
        out = torch.zeros_like(chi)
        i = torch.arange(n, device=DEV)
        for s, ks in zip(range(-9, 10), k):
            j = i + s
            j = (j.abs() - (j < 0).long()).clamp(max=2 * n - 1 - j) if dim == 1 else j % n   # reflect on the wall axis
            out.add_(chi.index_select(dim, j.clamp(0, n - 1)), alpha=float(ks))
        chi = out
    return _close_walls((1.0 - (1.0 - phi_min) * chi).clamp_(phi_min, 1.0))


class _Wave:
    """phi = 0.7 + amp sin(kx + a) cos(ky + b) sin(kz + c + 2 pi t/T) and its
    time derivative, evaluated on the device."""

    def __init__(self, shape, seed):
        g = _gen(seed)
        nx, ny, nz = shape
        self.amp = float(g.uniform(0.15, 0.2))
        a, b, c = g.uniform(0, 2 * math.pi, 3)

        def ang(n):
            return 2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n
        self.plane = (self.amp * torch.sin(ang(nx) + a).reshape(1, 1, nx)
                      * torch.cos(ang(ny) + b).reshape(1, ny, 1)).float()
        self.z = (ang(nz) + c).reshape(nz, 1, 1)
        self.mean = torch.full((1, 1, 1), 0.7, device=DEV)
        self.zero = torch.zeros((1, 1, 1), device=DEV)
        self.phi = torch.empty((nz, ny, nx), device=DEV)
        self.dphi = torch.empty((nz, ny, nx), device=DEV)

    def at(self, n):
        w = 2 * math.pi / WAVE_PERIOD
        ph = self.z + w * n
        torch.addcmul(self.mean, self.plane, torch.sin(ph).float(), out=self.phi)
        torch.addcmul(self.zero, self.plane, (w * torch.cos(ph)).float(), out=self.dphi)
        return self.phi, self.dphi


def _pulses(case, seed):
    """Snapshots (phi, d_t phi) of a pulsating product-sine bed at steps 0,
    10, 20, ...: the pulse closes after one pass."""
    shape = _shape(case)
    g = _gen(seed)
    ph = g.uniform(0, 2 * math.pi, 3)
    k = case["steps"] // STEPS_PER_REFRESH
    w = 2 * math.pi / case["steps"]
    bed = _sine("D3Q19", shape, 0.25, ph, torch.float64) - 0.05     # phi in [0.44, 0.96] with the pulse
    pulse = _sine("D3Q19", shape, 0.01, ph[::-1], torch.float64) - 0.99
    out = []
    for j in range(k):
        t = w * j * STEPS_PER_REFRESH
        out.append(((bed + pulse * math.sin(t)).float(), (pulse * (w * math.cos(t))).float()))
    return out


def _series(case, seed):
    """Per-step phi and force of a transient run (manufactured-solution
    pattern: smooth travelling fields), in the storage's field type."""
    nx, ny, nz = _shape(case)
    dim3 = nz > 1
    dt = torch.float64 if case["storage"] == "fp64" else torch.float32
    g = _gen(seed)
    ph = g.uniform(0, 2 * math.pi, (4, 3))
    amp = g.uniform(0.5e-5, 1e-5, 3)

    def field(p, t):
        s = [torch.sin(2 * math.pi * (torch.arange(n, dtype=torch.float64, device=DEV) + 0.01 * t) / n + q)
             for n, q in zip((nx, ny, nz), p)]
        f = s[0].reshape(1, 1, nx) * s[1].reshape(1, ny, 1)
        return f * s[2].reshape(nz, 1, 1) if dim3 else f.expand(nz, ny, nx)
    out = []
    for t in range(case["steps"]):
        phi = 0.5 + 0.4 * field(ph[0], t)
        force = torch.stack([a * field(q, t) for a, q in zip(amp, ph[1:])])
        if not dim3:
            force[2] = 0.0
        out.append((phi.to(dt).contiguous(), force.to(dt).contiguous()))
    p0 = (1e-4 * field(ph[1], 0)).to(dt).contiguous()
    u0 = torch.stack([1e-3 * field(q, 0) for q in ph[1:]]).to(dt).contiguous()
    if not dim3:
        u0[2] = 0.0
    return out, p0, u0


def _member_inputs(case, seed):
    """(lattice, shape, tau, phi) of every member of a batch."""
    g = _gen(seed)
    out = []
    for lattice, s in _members(case):
        shape = (s, s, s if lattice == "D3Q19" else 1)
        tau, amp = float(g.uniform(0.55, 1.2)), float(g.uniform(0.05, 0.3))
        phi = _sine(lattice, shape, amp, g.uniform(0, 2 * math.pi, 3), torch.float32)
        out.append((lattice, shape, tau, phi))
    return out


def _request_inputs(case, seed):
    """(LatticeSpec, phi on the host) of every request."""
    g = _gen(seed)
    out = []
    for j, (s, steps) in enumerate(_requests(case)):
        tau, amp = float(g.uniform(0.55, 1.2)), float(g.uniform(0.05, 0.3))
        phi = _sine("D3Q19", (s, s, s), amp, g.uniform(0, 2 * math.pi, 3), torch.float32).cpu().numpy()
        out.append((inputs.LatticeSpec("D3Q19", (s, s, s), tau, amp, j, steps=steps), phi))
    return out


def _solve_phi(case, seed):
    shape = _shape(case)
    dt = torch.float64 if case["storage"] == "fp64" else torch.float32
    g = _gen(seed)
    phi = _sine(case["lattice"], shape, float(g.uniform(0.1, 0.25)), g.uniform(0, 2 * math.pi, 3), dt)
    return _close_walls(phi) if _walls(case) else phi


DRAG = (150.0, 1.75, 6.0)     # Ergun constants, particle diameter in cells


# ------------------------------------------------------------ prepare and run

def _fields(n, f64):
    dt = torch.float64 if f64 else torch.float32
    return {"rho": torch.empty(n, dtype=dt, device=DEV), "p": torch.empty(n, dtype=dt, device=DEV),
            "u": torch.empty(3 * n, dtype=dt, device=DEV)}


def prepare(case, seed):
    kind, st = case["kind"], {"case": case}
    if kind == "batch":
        members = _member_inputs(case, seed)
        st["batch"] = lbm.Batch(max_members=len(members), storage=case["storage"])
        st["lats"] = []
        for lattice, shape, tau, phi in members:
            lat = lbm.Lattice(lattice, shape, tau=tau, storage=case["storage"])
            lat.set_epsilon(phi)
            lat.set_force((G, 0, 0))
            lat.init_equilibrium()
            st["batch"].add(lat, 10 ** 12)
            st["lats"].append(lat)
        st["out"] = _fields(sum(lat.n for lat in st["lats"]), False)
        return st
    if kind == "serve":
        st["server"] = serve.Server(storage=case["storage"], macro_steps=50, max_members=64, max_tiles=4096)
        st["requests"] = _request_inputs(case, seed)
        return st
    extra = {}
    if case.get("drag"):
        extra["drag"] = DRAG
    if case.get("les"):
        extra["les_cs"] = case["les"]
    lat = lbm.Lattice(case["lattice"], _shape(case), tau=case["tau"], storage=case["storage"], walls=_walls(case),
                      **extra)
    st["lat"], st["out"] = lat, _fields(lat.n, lat.f64)
    if kind == "solve":
        lat.set_epsilon(_solve_phi(case, seed))
    elif kind == "porous":
        lat.set_epsilon(_spheres(_shape(case), seed))
    elif kind == "wave":
        st["wave"] = _Wave(_shape(case), seed)
        lat.set_epsilon(*st["wave"].at(0))
    elif kind == "staged":
        st["snaps"] = [(e.cpu().reshape(-1).pin_memory(), d.cpu().reshape(-1).pin_memory())
                       for e, d in _pulses(case, seed)]
        st["host"] = [(e.numpy(), d.numpy()) for e, d in st["snaps"]]
        lat.set_epsilon(*st["host"][0])
    elif kind == "transient":
        st["series"], st["p0"], st["u0"] = _series(case, seed)
        lat.set_epsilon(st["series"][0][0])
    if kind != "transient":
        lat.set_force((G, 0, 0))
    lat.init_equilibrium()
    torch.cuda.synchronize()
    return st


def _read(lat, out):
    lat.moments_into(out["rho"], out["p"], out["u"])
    return out


def run(st):
    case = st["case"]
    kind, steps = case["kind"], case.get("steps", 0)
    if kind == "batch":
        st["batch"].step(steps, check=True)
        out, at = st["out"], 0
        mass = np.array([st["batch"].stats(lat)["mass"] for lat in st["lats"]])
        for lat in st["lats"]:
            n = lat.n
            lat.moments_into(out["rho"][at:at + n], out["p"][at:at + n], out["u"][3 * at:3 * (at + n)])
            at += n
        return {"fields": out, "mass": mass}
    if kind == "serve":
        reqs = [serve.Request(j, spec, 0.0, phi) for j, (spec, phi) in enumerate(st["requests"])]
        st["server"].run(reqs)
        st["server"].done.clear()
        return [r.result for r in reqs]
    lat = st["lat"]
    if kind == "solve":
        lat.init_equilibrium()
        stats = lat.step(steps)
    elif kind == "porous":
        stats = lat.step(steps)
    elif kind == "wave":
        for j in range(0, steps, STEPS_PER_REFRESH):
            n = lat.steps_done
            lat.set_epsilon(*st["wave"].at(n), n_ref=n)
            stats = lat.step(STEPS_PER_REFRESH, check_every=0 if j + STEPS_PER_REFRESH >= steps else -1)
    elif kind == "staged":
        snaps = st["host"]
        n = lat.steps_done
        lat.stage_epsilon(*snaps[0], n_ref=n)
        for j in range(len(snaps)):
            lat.commit_epsilon()
            if j + 1 < len(snaps):
                lat.stage_epsilon(*snaps[j + 1], n_ref=n + (j + 1) * STEPS_PER_REFRESH)
            stats = lat.step(STEPS_PER_REFRESH, check_every=0 if j + 1 == len(snaps) else -1)
    else:
        n = lat.steps_done
        lat.set_epsilon(st["series"][0][0], n_ref=n)
        lat.set_force((0, 0, 0), st["series"][0][1], n_ref=n)
        lat.init_equilibrium(p0=st["p0"], u0=st["u0"], integral=True, half_force=True)
        for j, (phi, force) in enumerate(st["series"]):
            lat.set_epsilon(phi, n_ref=n + j)
            lat.set_force((0, 0, 0), force, n_ref=n + j)
            stats = lat.step(1, check_every=0 if j + 1 == steps else -1)
    return {"fields": _read(lat, st["out"]), "mass": stats["mass"], "u_norm": stats["u_norm"]}


# --------------------------------------------------------------------- work

def _step_cost(lattice, elem, cells, steps, field_bytes):
    """One read and one write of every population and one read of the phi
    fields a step; about 20 operations per population."""
    q = Q_OF[lattice]
    return steps * cells * (2 * q * elem + field_bytes), steps * cells * 20.0 * q


def work(case):
    kind, elem = case["kind"], ELEM[case["storage"]]
    if kind == "batch":
        b = f = 0.0
        for lattice, s in _members(case):
            n = s ** (3 if lattice == "D3Q19" else 2)
            x = _step_cost(lattice, elem, n, case["steps"], 4)
            b, f = b + x[0] + n * (Q_OF[lattice] * elem + 24), f + x[1]
        return {"bytes": b, "flops": f}
    if kind == "serve":
        b = f = 0.0
        for s, steps in _requests(case):
            x = _step_cost("D3Q19", elem, s ** 3, steps, 4)
            b, f = b + x[0] + s ** 3 * (2 * 19 * elem + 24), f + x[1]
        return {"bytes": b, "flops": f}
    nx, ny, nz = _shape(case)
    n, q = nx * ny * nz, Q_OF[case["lattice"]]
    fe = 8 if case["storage"] == "fp64" else 4
    field = {"solve": fe, "porous": fe, "wave": 2 * fe, "staged": 2 * fe, "transient": 4 * fe}[kind]
    b, f = _step_cost(case["lattice"], elem, n, case["steps"], field)
    b += n * (q * elem + 6 * fe)                       # the moments: populations and phi in, rho, p, u out
    if kind in ("solve", "transient"):
        b += n * (q * elem + fe)                       # the initial state
    if kind in ("wave", "staged"):
        b += case["steps"] // STEPS_PER_REFRESH * n * 8    # the refreshed fields
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------ 64-bit restatement

class _Exact:
    """The scheme in plain torch float64: two arrays, pull streaming."""

    SETS = {"D1Q3": (1, {0: 2 / 3, 1: 1 / 6}), "D2Q9": (2, {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}),
            "D3Q19": (3, {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}),
            "D3Q27": (3, {0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216})}
    QUAD = {1: (1 / 2, 1 / 4), 2: (1 / 3, 1 / 6), 3: (1 / 6, 5 / 36)}

    def __init__(self, lattice, shape, tau, walls=0, drag=None, les=0.0):
        self.d, gw = self.SETS[lattice]
        c = [v for v in itertools.product((0, 1, -1), repeat=self.d) if sum(x * x for x in v) in gw]
        self.c = [v + (0,) * (3 - self.d) for v in c]
        self.w = [gw[sum(x * x for x in v)] for v in self.c]
        self.opp = [self.c.index(tuple(-x for x in v)) for v in self.c]
        self.tau, self.drag, self.les = tau, drag, les
        nx, ny, nz = shape
        self.shape = (nz, ny, nx)
        self.solid = torch.zeros(self.shape, dtype=torch.bool, device=DEV)
        if walls:
            self.solid[:, 0] = self.solid[:, -1] = True
        self.walls = walls
        self.g, self.field, self.n = (0.0, 0.0, 0.0), None, 0

    def set_phi(self, phi, dphi=None, n_ref=0):
        self.e = phi.reshape(self.shape).double()
        self.de = None if dphi is None else dphi.reshape(self.shape).double()
        self.n_ref = n_ref

    def phi(self):
        return self.e if self.de is None else self.e + (self.n - self.n_ref) * self.de

    def integral(self, e):
        w0, w1 = self.QUAD[self.d]
        return w0 * e + w1 * sum(torch.roll(e, s, 2 - a) for a in range(self.d) for s in (1, -1))

    def dot(self, i, v):
        s = 0.0
        for a in range(self.d):
            if self.c[i][a]:
                s = s + self.c[i][a] * v[a]
        return s

    def feq(self, i, m, u, usq):
        cu = self.dot(i, u)
        return self.w[i] * m * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)

    def init(self, p0=None, u0=None, integral=False, half_force=False):
        e = self.phi()
        rt = 1.0 if p0 is None else 1.0 + 3.0 * p0.reshape(self.shape).double()
        m = rt * (self.integral(e) if integral else e)
        zero = torch.zeros_like(e)
        u = [zero] * self.d if u0 is None else [u0.reshape((3,) + self.shape)[a].double() for a in range(self.d)]
        for k in range(2 if half_force else 1):
            usq = sum(x * x for x in u)
            self.f = [self.feq(i, m, u, usq) for i in range(len(self.w))]
            if half_force and k == 0:
                M0, _, F, _ = self.macro()
                u = [u[a] - 0.5 * F[a] / M0 for a in range(self.d)]

    def macro(self):
        f, e = self.f, self.phi()
        M0 = torch.zeros_like(e)
        J = [torch.zeros_like(e) for _ in range(self.d)]
        for i, fi in enumerate(f):
            M0 += fi
            for a in range(self.d):
                if self.c[i][a]:
                    J[a].add_(fi, alpha=self.c[i][a])
        rho = M0 / self.integral(e)
        F = []
        for a in range(self.d):
            grad = 0.5 * (torch.roll(e, -1, 2 - a) - torch.roll(e, 1, 2 - a))
            F.append(self.g[a] + rho / 3.0 * grad + (0.0 if self.field is None else self.field[a]))
        b = [J[a] + 0.5 * F[a] for a in range(self.d)]
        if self.drag is None:
            return M0, rho, F, [x / M0 for x in b]
        c1, c2, dp = self.drag
        lin = rho * c1 * (1.0 - e) ** 2 * ((self.tau - 0.5) / 3.0) / (e * dp * dp)
        quad = rho * c2 * (1.0 - e) / dp
        bn = torch.sqrt(sum(x * x for x in b))
        A = M0 + 0.5 * lin
        speed = 2.0 * bn / (A + torch.sqrt(A * A + 2.0 * quad * bn))
        u = [x / (A + 0.5 * quad * speed) for x in b]
        return M0, rho, [F[a] - (lin + quad * speed) * u[a] for a in range(self.d)], u

    def step(self, count):
        """Advance; the check sums (mass, |u|) are those of the last step's start."""
        for k in range(count):
            M0, rho, F, u = self.macro()
            usq = sum(x * x for x in u)
            uF = sum(u[a] * F[a] for a in range(self.d))
            if k + 1 == count:
                fluid = ~self.solid
                self.mass = float(M0[fluid].sum())
                self.u_norm = float(usq[fluid].sum().sqrt())
            tau = self.tau
            eq = None
            if self.les:
                eq = [self.feq(i, M0, u, usq) for i in range(len(self.w))]
                q2 = 0.0
                for a in range(self.d):
                    for b in range(self.d):
                        pab = sum(self.c[i][a] * self.c[i][b] * (self.f[i] - eq[i]) for i in range(len(self.w))
                                  if self.c[i][a] and self.c[i][b])
                        q2 = q2 + pab * pab
                tau = 0.5 * (tau + torch.sqrt(tau * tau + 18.0 * math.sqrt(2.0) * self.les ** 2
                                              * torch.sqrt(q2) / M0))
            cf, omega = 1.0 - 0.5 / tau, 1.0 / tau
            for i in range(len(self.w)):
                cF = self.dot(i, F)
                cu = self.dot(i, u)
                src = cf * self.w[i] * (3.0 * (cF - uF) + 9.0 * cu * cF)
                fe = eq[i] if eq is not None else self.feq(i, M0, u, usq)
                self.f[i] = self.f[i] + omega * (fe - self.f[i]) + src
            new = []
            for i, c in enumerate(self.c):
                x = torch.roll(self.f[i], (c[2], c[1], c[0]), (0, 1, 2)) if any(c) else self.f[i]
                if self.walls and c[1]:
                    # a population whose source is a wall layer returns from it
                    x = torch.where(torch.roll(self.solid, c[1], 1), self.f[self.opp[i]], x)
                new.append(x)
            if self.walls:
                for i in range(len(new)):
                    new[i] = torch.where(self.solid, torch.full_like(new[i], self.w[i]), new[i])
            self.f = new
            self.n += 1

    def fields(self):
        M0, rho, _, u = self.macro()
        u = torch.stack(u + [torch.zeros_like(rho)] * (3 - self.d))
        p = (rho - 1.0) / 3.0
        if self.walls:
            rho, p, u = (torch.where(self.solid, torch.zeros_like(x), x) for x in (rho, p, u))
        return {"rho": rho.reshape(-1), "p": p.reshape(-1), "u": u.reshape(-1)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        fields, mass = [], []
        for lattice, shape, tau, phi in _member_inputs(case, seed):
            x = _Exact(lattice, shape, tau)
            x.g = (G, 0.0, 0.0)
            x.set_phi(phi)
            x.init()
            x.step(case["steps"])
            fields.append(x.fields())
            mass.append(x.mass)
        return {"fields": {k: torch.cat([f[k] for f in fields]) for k in ("rho", "p", "u")}, "mass": np.array(mass)}
    if kind == "serve":
        out = []
        for spec, phi in _request_inputs(case, seed):
            s = spec.shape[0]
            x = _Exact("D3Q19", (s, s, s), spec.tau)
            x.g = (G, 0.0, 0.0)
            x.set_phi(torch.from_numpy(phi).to(DEV))
            x.init()
            x.step(spec.steps)
            f = x.fields()
            out.append({"u": f["u"].reshape(3, -1), "p": f["p"]})
        return out
    x = _Exact(case["lattice"], _shape(case), case["tau"], _walls(case), DRAG if case.get("drag") else None,
               case.get("les", 0.0))
    steps = case["steps"]
    if kind == "transient":
        series, p0, u0 = _series(case, seed)
        x.set_phi(series[0][0])
        x.field = series[0][1].double()
        x.init(p0, u0, integral=True, half_force=True)
        for phi, force in series:
            x.set_phi(phi)
            x.field = force.double()
            x.step(1)
    else:
        x.g = (G, 0.0, 0.0)
        if kind in ("solve", "porous"):
            x.set_phi(_solve_phi(case, seed) if kind == "solve" else _spheres(_shape(case), seed))
            x.init()
            x.step(steps)
        else:
            wave = _Wave(_shape(case), seed) if kind == "wave" else None
            snaps = None if wave else _pulses(case, seed)
            for n in range(0, steps, STEPS_PER_REFRESH):
                phi, dphi = wave.at(n) if wave else snaps[n // STEPS_PER_REFRESH]
                x.set_phi(phi, dphi, n)
                if n == 0:
                    x.init()
                x.step(STEPS_PER_REFRESH)
    return {"fields": x.fields(), "mass": x.mass, "u_norm": x.u_norm}
