"""The work that users of this package have it do, as cases that can be timed and checked.

A case is a dict of plain values.  ``prepare`` builds what a program holds before the call (a simulation, an
ensemble or an adjoint problem, set up from the seed and run in for a while), ``run`` is one pass through the public
entry points, ``work`` what the pass cannot do without, and ``exact`` the same pass in 64 bits with plain torch.

A pass of a single simulation rewinds it to its run-in state (a checkpoint in device memory), steps it and reads
fields and solid statistics.  Results are kept in the width of the simulation: float64 for fp64, float32 otherwise,
and bfloat16 (16 bits with the range that velocities need) for the vector fields of the two 16-bit storage variants.
"""
import math
import random  # noqa: F401  (draw takes a random.Random)

import numpy as np
import torch

KINDS = ("cavity", "settling", "mixing", "ellipses", "ensemble", "adjoint")
EPS, LAYERS, RMAX = 1.5, 11, 11
PHI_TIE, COS_TIE = 1e-9, 1e-9


def _case(name, kind, nx, ny, precision, solids, steps, spin, how="run", tile_x=32, tma=True, every=0):
    c = {"kind": kind, "nx": nx, "ny": ny, "precision": precision, "solids": solids, "steps": steps, "spin": spin,
         "how": how, "tile_x": tile_x, "tma": tma, "every": every}
    return {"name": name, **c} if name else c


def listed():
    return [
        # The smallest calls: a controller that advances one step at a time and looks at the disk after each, in
        # double precision, on the 64 x 64 cavity.  Latency and launches.
        _case("cavity64_f64_step_by_step", "cavity", 64, 64, "fp64", 1, 24, 8, how="calls"),
        # A whole run of a small cavity with one disk, as the coarse level of a grid-convergence study: one call,
        # hundreds of steps, a grid that fills a few of the chip's processors.
        _case("cavity80_f32", "cavity", 80, 80, "fp32", 1, 200, 50),
        # The middle level of that study on an odd grid (no tile shape divides it): one disk of radius 64.
        _case("cavity321_f32", "cavity", 321, 321, "fp32", 1, 100, 20),
        # The finest level: one disk of radius 128, the largest solid in use.
        _case("cavity640_f32", "cavity", 640, 640, "fp32", 1, 60, 10),
        # Two dozen heavy disks settling between walls: fewer solids than processors.
        _case("settling512_f32", "settling", 512, 512, "fp32", 24, 120, 30),
        # 506 ellipses in a closed box (the paper's 800 x 450 mixing): a non-disk level set on every node.
        _case("ellipses800x450_f32", "ellipses", 800, 450, "fp32", 506, 60, 20),
        # The benchmark workload with the launch configuration that the autotuner picks for it.
        _case("mixing4096_f32", "mixing", 4096, 4096, "fp32", 1024, 60, 30, tile_x=16, tma=False),
        # The same in 16-bit storage as a program gets it that leaves every option at its default.
        _case("mixing4096_f16", "mixing", 4096, 4096, "fp16", 1024, 40, 20),
        # A suspension on a ragged grid whose solid statistics are logged after every step into page-locked memory,
        # the way a program records trajectories without waiting for the device.
        _case("mixing1501x1203_f32_log", "mixing", 1501, 1203, "fp32", 110, 80, 20, how="log"),
        # The suspension in double precision, for reference solutions.
        _case("mixing1024_f64", "mixing", 1024, 1024, "fp64", 64, 30, 10),
        # An ensemble of 96 cavities of five sizes with one to eight disks each, advanced as one batch (parameter
        # sweeps); it runs on from pass to pass.
        _case("ensemble96_f32", "ensemble", 384, 384, "fp32", 96, 80, 10, tile_x=16),
        # Forward and backward: gradients of the disk's final position with respect to its materials and the body
        # force field, through the checkpointed reverse sweep (one iteration of a design loop).
        _case("adjoint256_f32", "adjoint", 256, 256, "fp32", 1, 160, 0, every=40),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("cavity", "cavity", "settling", "mixing", "mixing", "ellipses", "ensemble", "adjoint"))
    if kind == "cavity":
        n = _log_int(rng, 64, 640)
        precision = rng.choice(("fp32", "fp32", "fp64")) if n <= 200 else "fp32"
        how = rng.choice(("run", "run", "calls", "log"))
        steps = {"run": 100, "calls": 24, "log": 60}[how] if n <= 330 else 50
        return _case(None, kind, n, n, precision, 1, steps, rng.randint(5, 30), how, rng.choice((16, 32, 64)),
                     rng.random() < 0.5)
    if kind == "settling":
        nx, ny = _log_int(rng, 300, 900), _log_int(rng, 300, 900)
        return _case(None, kind, nx, ny, rng.choice(("fp32", "fp32", "fp16", "bf16")), max(6, nx * ny // 11000), 80,
                     rng.randint(5, 40), rng.choice(("run", "log")), rng.choice((16, 32, 64)), rng.random() < 0.5)
    if kind == "mixing":
        precision = rng.choice(("fp32", "fp32", "fp16", "bf16", "fp64"))
        hi = 1000 if precision == "fp64" else 4000
        nx, ny = _log_int(rng, 300, hi), _log_int(rng, 300, hi)
        return _case(None, kind, nx, ny, precision, max(4, nx * ny // 16384), 30 if precision == "fp64" else 40,
                     rng.randint(5, 30), rng.choice(("run", "run", "log")), rng.choice((16, 16, 32, 64, 128)),
                     rng.random() < 0.5)
    if kind == "ellipses":
        nx, ny = _log_int(rng, 200, 1000), _log_int(rng, 200, 700)
        return _case(None, kind, nx, ny, "fp32", max(1, (nx // 36) * (ny // 21)), 50, rng.randint(5, 30), "run",
                     rng.choice((16, 32)), rng.random() < 0.5)
    if kind == "ensemble":
        return _case(None, kind, rng.choice((256, 384)), 0, rng.choice(("fp32", "fp32", "fp16")), _log_int(rng, 4, 96),
                     60, 10, tile_x=rng.choice((16, 32)))
    n, steps = _log_int(rng, 96, 256), rng.randint(60, 160)
    return _case(None, "adjoint", n, n, rng.choice(("fp32", "fp32", "fp64")) if n < 160 else "fp32", 1, steps, 0,
                 every=rng.choice((25, 50, 100)))


# ---------------------------------------------------------------------------------------------------------------
# Inputs: geometry and materials from the seed
# ---------------------------------------------------------------------------------------------------------------


def _box(nx, ny, wall_x, wall_y, tau, **more):
    sc = {"name": "case", "nx": nx, "ny": ny, "wall_x": wall_x, "wall_y": wall_y, "tau": tau, "rho_f": 1.0,
          "lid_u": 0.0, "eps": EPS, "n_layers": LAYERS, "eta": 1.0, "gravity": 0.0, "force_kind": 0,
          "force_a": [0.0, 0.0], "solids": []}
    sc.update(more)
    return sc


def _place(rng, sc, count, r_lo, r_hi, rho, G, gap=4.0, keep=0.0):
    """Disks dropped at random, `gap` nodes from surface to surface and 3.5 nodes (+ keep) off a wall."""
    nx, ny = sc["nx"], sc["ny"]
    xs, ys, rs = np.zeros(count), np.zeros(count), np.zeros(count)
    n = 0
    for _ in range(count):
        r = rng.uniform(r_lo, r_hi)
        mx, my = (r + 3.5 + keep if sc[w] else 0.0 for w in ("wall_x", "wall_y"))
        for t in range(4000):
            if t % 200 == 199:  # no room for one of this size
                r *= 0.9
            x, y = rng.uniform(mx, nx - 1 - mx if mx else nx), rng.uniform(my, ny - 1 - my if my else ny)
            dx, dy = np.abs(xs[:n] - x), np.abs(ys[:n] - y)
            if not sc["wall_x"]:
                dx = np.minimum(dx, nx - dx)
            if not sc["wall_y"]:
                dy = np.minimum(dy, ny - dy)
            if np.all(np.hypot(dx, dy) >= rs[:n] + r + gap):
                xs[n], ys[n], rs[n] = x, y, r
                n += 1
                sc["solids"].append({"x": float(x), "y": float(y), "r": float(r), "rho_s": float(rng.uniform(*rho)),
                                     "G": float(rng.uniform(*G))})
                break
    return sc


def _cavity(case, rng):
    """A lid-driven cavity at Reynolds number 100 with a disk of radius L/5 in its middle."""
    L = case["nx"]
    U = 10.0 / L * rng.uniform(0.9, 1.0)
    sc = _box(L, L, 1, 1, 0.8, lid_u=U, deform_margin=0.6)
    sc["solids"].append({"x": L * rng.uniform(0.56, 0.62), "y": L * rng.uniform(0.47, 0.53),
                         "r": L * rng.uniform(0.195, 0.2), "rho_s": 1.0, "G": rng.uniform(0.08, 0.12) * U * U})
    return sc


def _ellipses(case, rng):
    """Lying and standing ellipses (semi-axes 8 x 4) on a jittered lattice, half of them heavy, under gravity."""
    nx, ny, n = case["nx"], case["ny"], case["solids"]
    cols = max(1, min(n, int(round(math.sqrt(n * nx / ny * 0.6)))))
    while cols > 1 and (nx - 23) / (cols - 1) < 20.5:
        cols -= 1
    if n == 506:
        cols = 23
    rows = -(-n // cols)
    sc = _box(nx, ny, 1, 1, 1.0, gravity=2e-5)
    for k in range(n):
        ix, iy = k % cols, k // cols
        x = 11.5 + ix * (nx - 24.0) / max(1, cols - 1) + rng.uniform(-0.5, 0.5)
        y = 11.5 + iy * (ny - 24.0) / max(1, rows - 1) + rng.uniform(-0.5, 0.5)
        lying = (ix + iy) % 2 == 0
        sc["solids"].append({"shape": "ellipse", "a": 8.0 if lying else 4.0, "b": 4.0 if lying else 8.0, "r": 8.0,
                             "x": float(x), "y": float(y), "rho_s": 1.25 if rng.random() < 0.48 else 0.83, "G": 0.05})
    return sc


def _vortex(sc):
    """Populations of a vortex that fills the cavity, at half the lid's speed: the flow that a run starts from."""
    n, U = sc["nx"], 0.5 * sc["lid_u"]
    p = np.pi * (np.arange(n) + 0.5) / n
    u = -U * np.sin(2 * p)[:, None] * np.sin(p)[None, :] ** 2
    v = U * np.sin(p)[:, None] ** 2 * np.sin(2 * p)[None, :]
    c = [CX[q] * u + CY[q] * v for q in range(9)]
    return np.stack([W[q] * (1 + 3 * c[q] + 4.5 * c[q] ** 2 - 1.5 * (u * u + v * v)) for q in range(9)])


def _smooth(rng, n, amp):
    y, x = np.mgrid[0:n, 0:n] / float(n)
    out = np.zeros((2, n, n))
    for c in range(2):
        for _ in range(3):
            kx, ky = rng.integers(1, 4, size=2)
            out[c] += rng.uniform(-amp, amp) * np.sin(2 * np.pi * (kx * x + ky * y) + rng.uniform(0, 2 * np.pi))
    return out


def _scenario(case, seed):
    rng = np.random.default_rng([KINDS.index(case["kind"]), case["nx"], case["ny"], int(seed)])
    kind, nx, ny = case["kind"], case["nx"], case["ny"]
    if kind == "cavity":
        return _cavity(case, rng)
    if kind == "settling":
        # packed closely enough for some blur zones (half-width 1.5) to overlap: contact
        return _place(rng, _box(nx, ny, 0, 1, 0.7, gravity=1e-5), case["solids"], 10, 20, (1.2, 2.0), (0.005, 0.02),
                      gap=2.0)
    if kind == "mixing":
        return _place(rng, _box(nx, ny, 0, 0, 0.6, force_kind=2, force_a=[1e-5, 0.0]), case["solids"], 8, 24,
                      (1.0, 1.5), (0.002, 0.02))
    if kind == "ellipses":
        return _ellipses(case, rng)
    if kind == "ensemble":
        sides = [s for s in (128, 192, 256, 384, 512) if s <= 2 * case["nx"] - 256]
        form, members = np.random.default_rng(case["solids"]), []  # the grids are the sweep's, whatever the seed
        for _ in range(case["solids"]):
            side, count = int(form.choice(sides)), int(form.integers(1, 9))
            sc = _box(side, side, 1, 1, 0.8, lid_u=float(rng.uniform(0.02, 0.03)))
            members.append(_place(rng, sc, count, 8, min(40.0, side / 8.0), (1.0, 1.0), (0.002, 0.01),
                                  keep=side / 16.0))
        return members
    n = nx
    sc = _box(n, n, 1, 1, 0.8, lid_u=float(rng.uniform(0.045, 0.05)), gravity=5e-5, force_kind=3)
    sc["solids"].append({"x": n * rng.uniform(0.58, 0.62), "y": n * rng.uniform(0.48, 0.52),
                         "r": n * rng.uniform(0.15, 0.157), "rho_s": float(rng.uniform(1.0, 1.1)),
                         "G": float(rng.uniform(0.008, 0.012))})
    sc["body_field"] = _smooth(rng, n, 5e-5)
    sc["dLdc"] = rng.uniform(0.5, 2.0, size=(1, 2))
    return sc


# ---------------------------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------------------------


def _kept(case):
    """Types in which vector fields, and scalars and statistics, are kept."""
    if case["precision"] == "fp64":
        return torch.float64, torch.float64
    return torch.float32 if case["precision"] == "fp32" else torch.bfloat16, torch.float32


def _fields(case, get, kept):
    """Density and velocity, and the cavity disk's level set or else the force density."""
    vector, scalar = kept
    out = {"rho": get("rho").to(scalar), "u": torch.stack([get("ux"), get("uy")]).to(vector)}
    if case["kind"] == "cavity":
        out["phi"] = get("phi").to(scalar)
    else:
        out["F"] = torch.stack([get("Fx"), get("Fy")]).to(vector)
    return out


def prepare(case, seed):
    import paper_2402_12696_gb300 as pkg
    sc = _scenario(case, seed)
    stream = torch.cuda.Stream()
    st = {"case": case, "stream": stream, "kept": _kept(case)}
    if case["kind"] == "ensemble":
        st["batch"] = pkg.Batch(sc, precision=case["precision"], stream=stream, tile_x=case["tile_x"])
        st["batch"].step(case["spin"])
        st["batch"].sync()
        return st
    sim = pkg.Simulation(sc, precision=case["precision"], stream=stream, tile_x=case["tile_x"], use_tma=case["tma"])
    st["sim"] = sim
    if case["kind"] == "adjoint":
        st["dLdc"] = sc["dLdc"]
        sim.init()
        return st
    if case["kind"] == "cavity":
        sim.init()
        sim.set_populations_host(_vortex(sc))
    sim.step(case["spin"])
    sim.sync()
    st["blob"] = sim.save()
    if case["how"] == "log":
        st["log"] = torch.zeros((case["steps"], sim.nsolids, 10), dtype=torch.float64).pin_memory()
    return st


def _split(stats, dtype):
    """Solid statistics: area, centroid, mass, momentum and deformation; the contact force on its own."""
    s = torch.as_tensor(stats).to(dtype)
    return {"solids": s[..., :8], "contact": s[..., 8:]}


def run(state):
    case, kept, stream = state["case"], state["kept"], state["stream"]
    vector, scalar = kept
    with torch.cuda.stream(stream):
        if case["kind"] == "ensemble":
            batch = state["batch"]
            batch.step(case["steps"])
            batch.sync()
            out = {"rho": torch.cat([m.field("rho").flatten().to(scalar) for m in batch.members]),
                   "u": torch.cat([m.field(f).flatten().to(vector) for f in ("ux", "uy") for m in batch.members])}
            out.update(_split(np.concatenate([m.solid_stats() for m in batch.members]), scalar))
            return out
        sim = state["sim"]
        if case["kind"] == "adjoint":
            c = sim.forward_checkpointed(case["steps"], case["every"])
            dG, dr, db = sim.backward(state["dLdc"], body=True)
            materials = torch.as_tensor(np.stack([dG, dr]))  # per solid, with respect to G and rho_s / rho_f
            return {"centroid": torch.as_tensor(c).to(scalar), "materials": materials.to(scalar), "body": db.to(vector)}
        sim.load(state["blob"])
        if case["how"] == "calls":
            seen = []
            for _ in range(case["steps"]):
                sim.step(1)
                seen.append(sim.solid_stats())
            host = lambda f: torch.as_tensor(sim.field_host(f))  # noqa: E731
            return {**_split(np.stack(seen), scalar), **_fields(case, host, kept)}
        if case["how"] == "log":
            import paper_2402_12696_gb300 as pkg
            log = state["log"]
            for k in range(case["steps"]):
                sim.step(1)
                pkg.lbrmt_solid_stats_async(sim.h, 0, log[k].data_ptr())
            out = _fields(case, sim.field, kept)
            sim.sync()
            return {**out, **_split(log, scalar)}
        sim.step(case["steps"])
        return {**_fields(case, sim.field, kept), **_split(sim.solid_stats(), scalar)}


def _mean_radius(case):
    return {"cavity": 0.1975 * case["nx"], "settling": 15.0, "mixing": 16.0, "ellipses": 6.0, "ensemble": 18.0,
            "adjoint": 0.1535 * case["nx"]}[case["kind"]]


def work(case):
    store = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case["precision"]]
    real = 8 if case["precision"] == "fp64" else 4
    nodes, solids = case["nx"] * case["ny"], case["solids"]
    if case["kind"] == "ensemble":
        nodes, solids = solids * 95000 * (1 if case["nx"] > 300 else 0.45), solids * 4.5
    band = solids * math.pi * (_mean_radius(case) + LAYERS) ** 2  # nodes that carry a reference map
    # per step: every population in and out; on the band the map in and out, the force out and in
    step_bytes = nodes * 18 * store + band * 6 * real
    # collision ~170 operations a node; advection, fits, stresses ~500 a band node
    step_flops = nodes * 170.0 + band * 500.0
    n, fields = case["steps"], {"ensemble": 3, "cavity": 4}.get(case["kind"], 5)
    if case["kind"] == "adjoint":  # forward, and the reverse step with its recorded state
        return {"bytes": n * (2 * step_bytes + nodes * 5 * 2 * real), "flops": n * 3 * step_flops}
    return {"bytes": n * step_bytes + nodes * (9 * store + fields * store), "flops": n * step_flops}


# ---------------------------------------------------------------------------------------------------------------
# The same pass in 64 bits: lattice Boltzmann with the reference map technique in plain torch
# ---------------------------------------------------------------------------------------------------------------

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _heaviside(p):
    h = 0.5 * (1 + p / EPS + torch.sin(math.pi * p / EPS) / math.pi)
    return torch.where(p <= -EPS, 0.0, torch.where(p >= EPS, 1.0, h))


def _sh(a, dy, dx):
    """a at the node (dy, dx) further on, in its own window (the windows' rims are never used)."""
    return torch.roll(a, (-dy, -dx), (-2, -1))


class _Plain:
    """One simulation: every solid has its own fixed window of the grid, all of one size."""

    def __init__(self, sc, travel):
        self.sc, dev = sc, "cuda" if torch.cuda.is_available() else "cpu"
        self.t = lambda v, d=torch.float64: torch.as_tensor(np.asarray(v), dtype=d, device=dev)
        so, nx, ny = sc["solids"], sc["nx"], sc["ny"]
        self.S, self.nx, self.ny, self.dev = len(so), nx, ny, dev
        col = lambda k: self.t([s[k] for s in so]).view(-1, 1, 1)  # noqa: E731
        self.xc, self.yc, self.R, self.rho_s, self.G = (col(k) for k in ("x", "y", "r", "rho_s", "G"))
        self.ell = bool(so) and "shape" in so[0]
        if self.ell:
            self.a, self.b = col("a"), col("b")
        half = int(math.ceil(max(s["r"] for s in so))) + LAYERS + 3 + travel
        T = self.T = 2 * half + 1
        self.ox, self.oy = (torch.floor(c).long() - half for c in (self.xc, self.yc))
        r = torch.arange(T, device=dev)
        self.gx, self.gy = (self.ox + r.view(1, 1, T)).expand(-1, T, T), (self.oy + r.view(1, T, 1)).expand(-1, T, T)
        one = torch.ones_like(self.gx, dtype=torch.bool)
        self.dom = one & (((self.gx >= 0) & (self.gx < nx)) if sc["wall_x"] else one)
        self.dom &= ((self.gy >= 0) & (self.gy < ny)) if sc["wall_y"] else one
        self.allowed = one & (((self.gx >= -2) & (self.gx <= nx + 1)) if sc["wall_x"] else one)
        self.allowed &= ((self.gy >= -2) & (self.gy <= ny + 1)) if sc["wall_y"] else one
        self.cell = (self.gy % ny) * nx + self.gx % nx
        ex, ey = (self.gx if sc["wall_x"] else self.gx % nx), (self.gy if sc["wall_y"] else self.gy % ny)
        self.eidx = ey.clamp(0, ny) * (nx + 1) + ex.clamp(0, nx)
        in_x, in_y = (ex >= 0) & (ex < nx), (ey >= 0) & (ey < ny)
        self.eok = (in_y & (ex >= 0) & (ex <= nx), in_x & (ey >= 0) & (ey <= ny))
        self._pairs()
        j = np.arange(ny)
        fb = np.zeros((2, ny, nx))
        if sc["force_kind"] == 2:
            fb[0] = (sc["force_a"][0] * np.sin(2 * np.pi * j / ny))[:, None]
        self.fb = self.t(sc["body_field"] if sc["force_kind"] == 3 else fb)
        self.start()

    def _pairs(self):
        """Pairs of solids that may come near each other, and where one's window lies in the other's."""
        sc, n = self.sc, self.S
        x, y, r = (v.flatten() for v in (self.xc, self.yc, self.R))
        dx, dy = (v[:, None] - v[None, :] for v in (x, y))
        if not sc["wall_x"]:
            dx = dx - self.nx * torch.round(dx / self.nx)
        if not sc["wall_y"]:
            dy = dy - self.ny * torch.round(dy / self.ny)
        near = torch.hypot(dx, dy) < r[:, None] + r[None, :] + 2 * EPS + 6
        near &= torch.ones(n, n, dtype=torch.bool, device=self.dev).triu(1)
        self.ps, self.pt = torch.nonzero(near, as_tuple=True)

    def phi0(self, X, Y):
        qx, qy = X - self.xc, Y - self.yc
        if not self.ell:
            return torch.sqrt(qx * qx + qy * qy) - self.R
        tall = self.a < self.b
        e0, e1 = torch.maximum(self.a, self.b), torch.minimum(self.a, self.b)
        y0, y1 = torch.where(tall, qy, qx).abs(), torch.where(tall, qx, qy).abs()
        z0, z1, r0 = y0 / e0, y1 / e1, (e0 / e1) ** 2
        n0 = r0 * z0
        g = z0 * z0 + z1 * z1 - 1
        lo, hi = z1 - 1, torch.where(g < 0, 0.0, torch.hypot(n0, z1) - 1)
        s = lo.clone()
        for _ in range(40):  # Newton from the left end of the bracket: monotone on a convex function
            ia, ib = 1 / (s + r0), 1 / (s + 1).clamp_min(1e-300)
            f = (n0 * ia) ** 2 + (z1 * ib) ** 2 - 1
            s = torch.minimum(torch.maximum(s, s + f / (2 * ((n0 * ia) ** 2 * ia + (z1 * ib) ** 2 * ib))), hi)
            s = torch.where(torch.isfinite(s), s, lo)
        d = torch.hypot(r0 * y0 / (s + r0) - y0, y1 / (s + 1) - y1)
        x = (e0 * y0 / (e0 * e0 - e1 * e1)).clamp(max=1)
        on0 = torch.hypot(e0 * x - y0, e1 * torch.sqrt(1 - x * x))
        on0 = torch.where(e0 * y0 < e0 * e0 - e1 * e1, on0, (y0 - e0).abs())
        d = torch.where(y1 > 0, torch.where(y0 > 0, d, (y1 - e1).abs()), on0)
        return torch.where(g < 0, -d, d)

    def start(self):
        X, Y = self.gx.double(), self.gy.double()
        S = self.dom & (self.phi0(X, Y) < -PHI_TIE)
        self.lab = self.layers(S)
        keep = self.lab >= 0
        self.X, self.Y = torch.where(keep, X, 0.0), torch.where(keep, Y, 0.0)
        self.phi = self.phi0(self.X, self.Y)
        _, _, drho = self.force()
        w = torch.tensor(W, dtype=torch.float64, device=self.dev).view(9, 1, 1)
        self.f = w * torch.ones_like(drho)
        self.f = torch.cat([self.f[:1] + drho, self.f[1:]])
        self.moments(0.0, 0.0)

    def moments(self, hx, hy):
        """Density and velocity, with half of the momentum (hx, hy) that the force brings in a step."""
        f = self.f
        self.rho = r = f.sum(0)
        self.ux = (f[1] - f[3] + f[5] - f[6] + f[8] - f[7] + 0.5 * hx) / r
        self.uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8] + 0.5 * hy) / r

    def layers(self, S):
        lab = torch.where(S, 0, -1).to(torch.int8)
        for k in range(1, LAYERS + 1):
            on = lab == k - 1
            near = _sh(on, 1, 0) | _sh(on, -1, 0) | _sh(on, 0, 1) | _sh(on, 0, -1)
            lab = torch.where(near & (lab < 0) & self.allowed, torch.tensor(k, dtype=torch.int8, device=self.dev), lab)
        return lab

    def fit(self, l, X, Y, lab, old):
        """Values of layer l from the weighted plane fits of the nodes before it."""
        T = self.T
        t = torch.nonzero(lab.flatten() == l).flatten()
        ty, tx = (t // T) % T, t % T
        use, nhx, nhy = None, None, None
        if l <= 2:
            phi, ok = old
            n4 = [(1, 0), (-1, 0), (0, 1), (0, -1)]
            use = torch.stack([ok.flatten()[t + dx + dy * T] for dx, dy in n4]).all(0)
            e, w, n, s = (phi.flatten()[t + dx + dy * T] for dx, dy in n4)
            gx, gy = (e - w) / 2, (n - s) / 2
            nn = torch.sqrt(torch.where(use, gx * gx + gy * gy, 1.0))
            use = use & (nn > 0)
            nhx, nhy = (torch.where(use, g / torch.where(nn > 0, nn, 1.0), 0.0) for g in (gx, gy))
        done = torch.zeros_like(t, dtype=torch.bool)
        vx, vy = torch.zeros_like(t, dtype=torch.float64), torch.zeros_like(t, dtype=torch.float64)
        left = torch.arange(len(t), device=self.dev)
        for r in range(2, RMAX + 1):
            d = torch.arange(-r, r + 1, device=self.dev)
            dx, dy = d.repeat(2 * r + 1), d.repeat_interleave(2 * r + 1)
            mid = (dx != 0) | (dy != 0)
            dx, dy = dx[mid], dy[mid]
            x, y = tx[left, None] + dx, ty[left, None] + dy
            inside = (x >= 0) & (x < T) & (y >= 0) & (y < T)
            k = torch.where(inside, t[left, None] + dy * T + dx, t[left, None])
            L = lab.flatten()[k]
            valid = inside & (L >= 0) & (L < l)
            w = torch.where(valid, 2.0 ** -(dx.abs() + dy.abs()).double(), 0.0)
            if use is not None:
                c = (-dx * nhx[left, None] - dy * nhy[left, None]) / torch.hypot(dx.double(), dy.double())
                w = torch.where(use[left, None], torch.where(c > COS_TIE, c * w, 0.0), w)
            pos = w > 0
            n = pos.sum(1)
            sx, sy = (pos * dx).sum(1), (pos * dy).sum(1)
            sxx, syy, sxy = (pos * dx * dx).sum(1), (pos * dy * dy).sum(1), (pos * dx * dy).sum(1)
            gram = (n * sxx - sx * sx) * (n * syy - sy * sy) - (n * sxy - sx * sy) ** 2
            fx, fy = dx.double(), dy.double()
            a, b, c, e, g, h = ((w * q).sum(1) for q in (fx * fx, fx * fy, fx, fy * fy, fy, torch.ones_like(fx)))
            det = a * (e * h - g * g) - b * (b * h - c * g) + c * (b * g - c * e)
            ok = (valid.sum(1) >= 3) & (n >= 3) & (gram != 0) & (det != 0)
            c13, c23, c33 = b * g - c * e, b * c - a * g, a * e - b * b
            coef = w * (c13[:, None] * fx + c23[:, None] * fy + c33[:, None]) / torch.where(ok, det, 1.0)[:, None]
            x0, y0 = self.gx.flatten()[t[left]].double(), self.gy.flatten()[t[left]].double()
            got = left[ok]
            px = x0 + (coef * (X.flatten()[k] - x0[:, None])).sum(1)
            py = y0 + (coef * (Y.flatten()[k] - y0[:, None])).sum(1)
            vx, vy = vx.index_put((got,), px[ok]), vy.index_put((got,), py[ok])
            done[got] = True
            left = torch.nonzero(~done).flatten()
            if not len(left):
                break
        shape = X.shape
        return X.flatten().index_put((t,), vx).view(shape), Y.flatten().index_put((t,), vy).view(shape)

    def advect(self):
        u, v = self.ux.flatten()[self.cell], self.uy.flatten()[self.cell]
        S = self.dom & (self.lab >= 0) & (self.phi < -PHI_TIE)
        back, down = u >= 0, v >= 0
        new = []
        for A in (self.X, self.Y):
            side = lambda y, x: (3 * A - 4 * _sh(A, y, x) + _sh(A, 2 * y, 2 * x)) / 2  # noqa: E731, B023
            dx = torch.where(back, side(0, -1), -side(0, 1))
            dy = torch.where(down, side(-1, 0), -side(1, 0))
            new.append(torch.where(S, A - (u * dx + v * dy), 0.0))
        lab = self.layers(S)
        old = (self.phi, self.lab >= 0)
        X, Y = new
        for l in range(1, LAYERS + 1):
            X, Y = self.fit(l, X, Y, lab, old)
        self.X, self.Y, self.lab = X, Y, lab
        self.phi = torch.where(lab >= 0, self.phi0(torch.where(lab >= 0, X, self.gx.double()),
                                                   torch.where(lab >= 0, Y, self.gy.double())), 99.0)

    def edges(self, d, A):
        """Derivatives across and along the half-edges of direction d, and the edge mean."""
        if d == 0:
            lo = lambda k: _sh(A, k, -1)  # noqa: E731
            hi = lambda k: _sh(A, k, 0)  # noqa: E731
        else:
            lo = lambda k: _sh(A, -1, k)  # noqa: E731
            hi = lambda k: _sh(A, 0, k)  # noqa: E731
        return hi(0) - lo(0), (hi(1) + lo(1) - hi(-1) - lo(-1)) / 4, (hi(0) + lo(0)) / 2

    @staticmethod
    def whole(d, ok):
        """Are all six nodes of the half-edge's stencil in the band?"""
        both = ok & (_sh(ok, 0, -1) if d == 0 else _sh(ok, -1, 0))
        return both & (_sh(both, 1, 0) & _sh(both, -1, 0) if d == 0 else _sh(both, 0, 1) & _sh(both, 0, -1))

    def force(self):
        nx, ny, sc, ok = self.nx, self.ny, self.sc, self.lab >= 0
        NE, tau = (nx + 1) * (ny + 1), []
        zero = lambda n: torch.zeros(n, dtype=torch.float64, device=self.dev)  # noqa: E731
        for d in (0, 1):
            Xn, Xt, _ = self.edges(d, self.X - self.gx)
            Yn, Yt, _ = self.edges(d, self.Y - self.gy)
            _, _, ph = self.edges(d, self.phi)
            on = self.whole(d, ok) & self.eok[d] & (ph < EPS)
            Axx, Axy, Ayx, Ayy = (Xn, Xt, Yn, Yt) if d == 0 else (Xt, Xn, Yt, Yn)
            Axx, Axy, Ayx, Ayy = (torch.where(on, q, 0.0) for q in (Axx, Axy, Ayx, Ayy))
            det = (1 + Axx) * (1 + Ayy) - Axy * Ayx
            Fxx, Fxy, Fyx, Fyy = (1 + Ayy) / det, -Axy / det, -Ayx / det, (1 + Axx) / det
            Bxx, Bxy, Byy = Fxx * Fxx + Fxy * Fxy, Fxx * Fyx + Fxy * Fyy, Fyx * Fyx + Fyy * Fyy
            tr = (Bxx + Byy + 1) / 3
            lam = torch.where(on, 1 - _heaviside(torch.where(on, ph, 0.0)), 0.0)
            at = self.eidx[on]
            put = lambda q: zero(NE).index_add(0, at, q[on])  # noqa: E731
            L = put(lam)
            s = [put(lam * self.G * q) for q in (Bxx - tr, Bxy, Byy - tr)]
            s = [q / torch.where(L > 1, L, 1.0) for q in s]
            tau.append([q + k for q, k in zip(s, self.contact(d, ok))])
        lam = torch.where(ok & self.dom, 1 - _heaviside(self.phi), 0.0)
        on = lam > 0
        node = lambda q: zero(nx * ny).index_add(0, self.cell[on], (lam * q)[on]).view(ny, nx)  # noqa: E731
        L = node(torch.ones_like(lam))
        L = torch.where(L > 1, L, 1.0)
        drho = node((self.rho_s - 1.0).expand_as(lam)) / L
        acc = node((-(1 - 1.0 / self.rho_s) * sc["gravity"]).expand_as(lam)) / L if sc["gravity"] else 0.0
        i, j = torch.arange(nx, device=self.dev), torch.arange(ny, device=self.dev)
        i1, j1 = (i + 1) if sc["wall_x"] else (i + 1) % nx, (j + 1) if sc["wall_y"] else (j + 1) % ny
        x, y = ([q.view(ny + 1, nx + 1) for q in tau[d]] for d in (0, 1))
        rt = lambda q: q[:ny][:, i1] - q[:ny][:, i]  # noqa: E731
        up = lambda q: q[j1][:, :nx] - q[j][:, :nx]  # noqa: E731
        return rt(x[0]) + up(y[1]) + self.fb[0], rt(x[1]) + up(y[2]) + acc + self.fb[1], drho

    def contact(self, d, ok):
        sc, T, out = self.sc, self.T, []
        NE = (self.nx + 1) * (self.ny + 1)
        total = [torch.zeros(NE, dtype=torch.float64, device=self.dev) for _ in range(3)]
        for k in range(0, len(self.ps), 256):
            s, t = self.ps[k:k + 256], self.pt[k:k + 256]
            sx, sy = self.ox[s] - self.ox[t], self.oy[s] - self.oy[t]
            if not sc["wall_x"]:
                sx = sx - self.nx * torch.round(sx / self.nx).long()
            if not sc["wall_y"]:
                sy = sy - self.ny * torch.round(sy / self.ny).long()
            r = torch.arange(T, device=self.dev)
            lx, ly = r.view(1, 1, T) + sx, r.view(1, T, 1) + sy
            inside = (lx >= 0) & (lx < T) & (ly >= 0) & (ly < T)
            at = t.view(-1, 1, 1) * T * T + ly.clamp(0, T - 1) * T + lx.clamp(0, T - 1)
            okt, pt = ok.flatten()[at] & inside, self.phi.flatten()[at]
            _, _, es = self.edges(d, self.phi[s])
            _, _, et = self.edges(d, pt)
            on = self.whole(d, ok[s]) & self.whole(d, okt) & self.eok[d][s] & (es < EPS) & (et < EPS)
            if not bool(on.any()):
                continue
            gn, gt, _ = self.edges(d, self.phi[s] - pt)
            gx, gy = (gn, gt) if d == 0 else (gt, gn)
            gx, gy = gx[on], gy[on]
            nn = torch.sqrt(gx * gx + gy * gy)
            nx_, ny_ = gx / torch.where(nn > 0, nn, 1.0), gy / torch.where(nn > 0, nn, 1.0)
            f = torch.minimum(0.5 * (1 - es[on] / EPS), 0.5 * (1 - et[on] / EPS))
            kk = -sc["eta"] * f * (self.G[s] + self.G[t]).expand_as(on)[on] * (nn > 0)
            for q, v in enumerate((kk * (nx_ * nx_ - 0.5), kk * nx_ * ny_, kk * (ny_ * ny_ - 0.5))):
                total[q] = total[q].index_add(0, self.eidx[s][on], v)
        return total

    def fluid(self, Fx, Fy, drho):
        sc, nx, ny = self.sc, self.nx, self.ny
        om, kf = 1 / sc["tau"], 1 - 0.5 / sc["tau"]
        rho, u, v, fh = self.rho, self.ux, self.uy, []
        uu, uF = u * u + v * v, u * Fx + v * Fy
        for q in range(9):
            cu, cF = CX[q] * u + CY[q] * v, CX[q] * Fx + CY[q] * Fy
            eq = W[q] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu) + ((1 - W[0]) if q == 0 else -W[q]) * drho
            fh.append(self.f[q] - om * (self.f[q] - eq) + kf * rho * W[q] * (3 * (cF - uF) + 9 * cu * cF))
        new = []
        for q in range(9):
            a = torch.roll(fh[q], (CY[q], CX[q]), (0, 1))
            if (sc["wall_x"] and CX[q]) or (sc["wall_y"] and CY[q]):
                wall = torch.zeros(ny, nx, dtype=torch.bool, device=self.dev)
                lid = torch.zeros_like(wall)
                if sc["wall_x"] and CX[q]:
                    wall[:, 0 if CX[q] > 0 else nx - 1] = True
                if sc["wall_y"] and CY[q]:
                    wall[0 if CY[q] > 0 else ny - 1] = True
                    if CY[q] < 0:
                        lid[ny - 1] = True
                a = torch.where(wall, fh[OPP[q]] + 6 * W[q] * rho * CX[q] * sc["lid_u"] * lid, a)
            new.append(a)
        self.f = torch.stack(new)
        self.moments(rho * Fx, rho * Fy)

    def step(self):
        self.advect()
        self.Fx, self.Fy, drho = self.force()
        self.fluid(self.Fx, self.Fy, drho)

    def sums(self):
        lam = torch.where((self.lab >= 0) & self.dom, 1 - _heaviside(self.phi), 0.0)
        tot = lambda q: (lam * q).sum((1, 2))  # noqa: E731
        A = tot(torch.ones_like(lam))
        return lam, tot, A, tot(self.gx.double()) / A, tot(self.gy.double()) / A

    def stats(self):
        lam, tot, A, cx, cy = self.sums()
        rho, u, v = (q.flatten()[self.cell] for q in (self.rho, self.ux, self.uy))
        ok = self.lab >= 0
        on = ok & self.dom & (self.phi < -PHI_TIE)
        on = on & _sh(ok, 0, 1) & _sh(ok, 0, -1) & _sh(ok, 1, 0) & _sh(ok, -1, 0)
        D = lambda B, dy, dx: (_sh(B, dy, dx) - _sh(B, -dy, -dx)) / 2  # noqa: E731
        ex, ey = self.X - self.gx, self.Y - self.gy
        xx, xy, yx, yy = D(ex, 0, 1), D(ex, 1, 0), D(ey, 0, 1), D(ey, 1, 0)
        dl = xx + yy + xx * yy - xy * yx
        dev = torch.where(on, (dl / (1 + dl)).abs(), 0.0)
        lon = torch.where(on, lam, 0.0)
        mean = (lon * dev).sum((1, 2)) / lon.sum((1, 2))
        return torch.stack([A, cx, cy, tot(rho), tot(rho * u), tot(rho * v), dev.amax((1, 2)), mean], 1)


def _plain_pass(sc, case):
    m = _Plain(sc, 4)
    if case["kind"] == "cavity":
        m.f = m.t(_vortex(sc))
        m.moments(0.0, 0.0)
    for _ in range(case["spin"]):
        m.step()
    seen = []
    for _ in range(case["steps"]):
        m.step()
        if case["how"] != "run":
            seen.append(m.stats())
    out = {"rho": m.rho, "u": torch.stack([m.ux, m.uy])}
    if case["kind"] == "cavity":
        on = (m.lab >= 0) & m.dom
        out["phi"] = torch.full_like(m.rho, math.nan).flatten().index_put((m.cell[on],), m.phi[on]).view_as(m.rho)
    else:
        out["F"] = torch.stack([m.Fx, m.Fy])
    return {**out, "solids": torch.stack(seen) if seen else m.stats()}


def exact(case, seed):
    sc = _scenario(case, seed)
    if case["kind"] == "adjoint":
        m = _Plain(sc, 4)
        G, ratio = m.G.clone().requires_grad_(), m.rho_s.clone().requires_grad_()
        body = m.fb.clone().requires_grad_()
        m.G, m.rho_s, m.fb = G, ratio, body
        m.start()
        for _ in range(case["steps"]):
            m.step()
        _, _, _, cx, cy = m.sums()
        c = torch.stack([cx, cy], 1)
        g = torch.autograd.grad((c * m.t(sc["dLdc"])).sum(), (G, ratio, body))
        return {"centroid": c.detach(), "materials": torch.stack([g[0].flatten(), g[1].flatten()]), "body": g[2]}
    with torch.no_grad():
        if case["kind"] == "ensemble":
            if case["solids"] > 10:  # half a minute and more of plain torch
                return None
            parts = [_plain_pass(s, case) for s in sc]
            out = {"rho": torch.cat([p["rho"].flatten() for p in parts]),
                   "u": torch.cat([p["u"][k].flatten() for k in (0, 1) for p in parts]),
                   "solids": torch.cat([p["solids"] for p in parts])}
        else:
            out = _plain_pass(sc, case)
        return {**out, "contact": None}
