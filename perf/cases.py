"""The workloads whose time matters to users of this package, as cases that can be timed and checked.

A case is a dict of plain values.  `prepare` makes what a program holds before the call (the lattice handle, the
state it resumes from, the output buffers), `run` makes one pass through the public entry points, `work` says what
a pass cannot do without, and `exact` states the same computation in plain torch and 64 bits.

Kinds:
  advance2d / advance3d  resume a checkpointed flow (load_state), advance it, and save it again with its fields
  loop2d / loop3d        the design loop: from rest, a first solve and a few {exchange, re-solve} iterations
  batch                  candidate distributors stepped together: a solve, an exchange and a re-solve of each
  served                 a burst of requests into the request loop (solves, and whole optimisations)
"""
import functools
import itertools
import math
import random

import numpy as np
import torch

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

STORAGE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
COLLISION = {"bgk": L.COLLIDE_BGK, "regularized": L.COLLIDE_REGULARIZED, "smagorinsky": L.COLLIDE_SMAGORINSKY}
C_SMAG = 0.1
# floating-point operations of one cell update: moments, equilibria, relaxation, closure
FLOPS2, FLOPS3 = 130, 330


def listed():
    return [
        # The shortest call: a 128 x 64 T-junction advanced by a hundred steps between two looks at its fields.
        dict(name="junction_advance", kind="advance2d", geometry="junction", tau=0.8, u_max=0.05, steps=100,
             precision="f32", collision="bgk"),
        # The smallest design loop, configs/t_junction_128x64.json: solves of 2000 steps, an exchange before each.
        dict(name="junction_loop", kind="loop2d", geometry="junction", tau=0.8, u_max=0.05, steps=2000, iters=2,
             precision="f32", collision="bgk"),
        # configs/tree_2048x1024_g4.json: the full-size distributor, 16 outlets, 0.2 % of the fluid exchanged.
        dict(name="tree_loop_f32", kind="loop2d", geometry="tree2048", tau=0.53, u_max=0.01171875, steps=2000,
             iters=2, precision="f32", collision="bgk"),
        # configs/tree_2048x1024_g4_16bit.json: the same with 16-bit populations.
        dict(name="tree_loop_bf16", kind="loop2d", geometry="tree2048", tau=0.53, u_max=0.01171875, steps=2000,
             iters=2, precision="bf16", collision="bgk"),
        # The collector on a half domain (a symmetry plane below row 0): small, thousands of steps a solve.
        dict(name="collector_loop", kind="loop2d", geometry="collector", tau=0.53, u_max=0.03, steps=5000, iters=2,
             precision="f32", collision="bgk"),
        # A distributor of odd size with the eddy-viscosity model that higher Reynolds numbers need.
        dict(name="smagorinsky_advance", kind="advance2d", geometry="tree", nx=1501, ny=751, generations=4, w0=46,
             geo_seed=3, tau=0.53, u_max=0.0163, steps=2000, precision="f32", collision="smagorinsky"),
        # A wide channel array far beyond the L2 cache, and one of odd size with 16-bit populations.
        dict(name="channels_f32", kind="advance2d", geometry="channels", nx=8192, ny=4096, channels=16, tau=0.6,
             u_max=0.05, steps=256, precision="f32", collision="bgk"),
        dict(name="channels_bf16", kind="advance2d", geometry="channels", nx=7001, ny=3501, channels=16, tau=0.6,
             u_max=0.05, steps=256, precision="bf16", collision="bgk"),
        # configs/candidates_256.json: uneven candidate distributors in one batch, both storage types.
        dict(name="candidates_f32", kind="batch", n=256, geo_seed=0, steps=500, precision="f32"),
        dict(name="candidates_bf16", kind="batch", n=256, geo_seed=0, steps=500, precision="bf16"),
        # The D3Q19 distributor of 384 x 192 x 192 cells.
        dict(name="tree3d_advance", kind="advance3d", geometry="tree3d", nx=384, ny=192, nz=192, generations=4, w0=48,
             tau=0.53, u_max=0.0234375, steps=200, precision="f32", collision="bgk"),
        # configs/served_poisson_200.json: a burst of mixed requests, solves and optimisations of 128 to 2048 cells.
        dict(name="served_burst", kind="served", n=16, geo_seed=100, steps=1000, precision="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _tree_case(rng, lo, hi):
    nx = _log(rng, lo, hi)
    ny = nx // 2
    g = min(4, max(1, int(math.log2(nx / 128.0)) + 1))
    w0 = max(8, ny // 16)
    return dict(geometry="tree", nx=nx, ny=ny, generations=g, w0=w0, geo_seed=rng.randrange(1000), tau=0.53,
                u_max=min(0.05, 0.75 / w0))


def draw(rng):
    """One more case of the listed ranges: sizes spread over their logarithm, odd ones among them."""
    kind = rng.choice(["advance2d", "advance2d", "advance2d", "loop2d", "loop2d", "batch", "advance3d", "loop3d",
                       "served"])
    precision = rng.choice(["f32", "f32", "bf16", "f16"])
    if kind == "advance2d":
        c = dict(kind=kind, steps=2 * _log(rng, 50, 500), precision=precision,
                 collision=rng.choice(["bgk", "bgk", "bgk", "regularized", "smagorinsky"]))
        if rng.random() < 0.5:
            c.update(_tree_case(rng, 128, 2048))
        else:
            nx = _log(rng, 1000, 8192)
            c.update(geometry="channels", nx=nx, ny=nx // 2 + rng.randrange(2), channels=rng.choice([4, 8, 16]),
                     tau=0.6, u_max=0.05, collision="bgk", steps=2 * _log(rng, 50, 150))
        return c
    if kind == "loop2d":
        return dict(kind=kind, steps=2 * _log(rng, 100, 1000), iters=rng.randrange(1, 4), precision=precision,
                    collision="bgk", **_tree_case(rng, 128, 2048))
    if kind == "batch":
        return dict(kind=kind, n=_log(rng, 8, 128), geo_seed=rng.randrange(1000), steps=2 * _log(rng, 50, 250),
                    precision=precision)
    if kind == "served":
        return dict(kind=kind, n=_log(rng, 4, 16), geo_seed=rng.randrange(1000), steps=1000, precision=precision)
    nx = _log(rng, 72, 320)
    if rng.random() < 0.5:
        c = dict(geometry="tree3d", nx=nx, ny=nx // 2, nz=nx // 2, generations=2 if nx < 160 else 4,
                 w0=max(10, nx // 8), tau=0.53, u_max=min(0.05, 1.125 / max(10, nx // 8)))
    else:
        c = dict(geometry="duct3d", nx=nx, ny=nx // 2, nz=nx // 2 - rng.randrange(3), tau=0.6, u_max=0.05)
    c.update(kind=kind, steps=2 * _log(rng, 25, 100), precision=precision,
             collision=rng.choice(["bgk", "bgk", "smagorinsky"]))
    if kind == "loop3d":
        c.update(collision="bgk", iters=1, geometry="tree3d", generations=2 if nx < 160 else 4, w0=max(10, nx // 8),
                 ny=nx // 2, nz=nx // 2, tau=0.53, u_max=min(0.05, 1.125 / max(10, nx // 8)))
    return c


# ---- geometry ------------------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _cells_of(key):
    c = dict(key)
    g = c["geometry"]
    if g == "junction":
        return I.config_t_junction()["cells"]
    if g == "tree2048":
        return I.config_tree_2048()["cells"]
    if g == "collector":
        return I.config_collector()["cells"]
    if g == "tree":
        return I.tree(c["nx"], c["ny"], c["generations"], c["w0"], seed=c["geo_seed"])
    if g == "channels":
        return I.channel_array(c["nx"], c["ny"], c["channels"])
    if g == "tree3d":
        return I.tree3d(c["nx"], c["ny"], c["nz"], c["generations"], c["w0"])
    return I.duct3d(c["nx"], c["ny"] - 2, c["nz"] - 2)


def _cells(case):
    keep = ("geometry", "nx", "ny", "nz", "generations", "w0", "geo_seed", "channels")
    return _cells_of(tuple((k, case[k]) for k in keep if k in case))


@functools.lru_cache(maxsize=2)
def _candidates(n, geo_seed):
    return I.config_candidates(n, geo_seed)


@functools.lru_cache(maxsize=2)
def _requests(n, geo_seed):
    return [I.config_served_request(geo_seed + k) for k in range(n)]


def _fluid(cells):
    return int(cells.size - np.count_nonzero(cells))


def _u_max(case, seed):
    """The inlet speed of the case, within a tenth: the design points of a program differ in it."""
    return case["u_max"] * (0.9 + 0.2 * random.Random(seed).random())


# ---- the velocity sets, for making a state and for the 64-bit statement --------------------------------------------

C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
      (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
      (0, -1, 1)]
W3 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _state(cells, seed, u_max, dtype):
    """A developed flow to resume from, as a checkpoint holds it: shifted populations of smooth density and velocity
    fields (a few random waves about a stream along x), zero on solid cells."""
    dims = cells.ndim
    c, w = (C2, W2) if dims == 2 else (C3, W3)
    r = random.Random(seed)
    dev = "cuda"
    axes = [torch.arange(n, device=dev, dtype=torch.float32) / n for n in cells.shape]
    fluid = torch.from_numpy(cells).to(dev) == 0

    def waves(amplitude):
        f = torch.zeros(cells.shape, device=dev)
        for _ in range(3):
            term = torch.ones((), device=dev)
            for a, x in enumerate(axes):
                shape = [1] * dims
                shape[a] = -1
                term = term * torch.cos(2 * math.pi * (r.randrange(1, 5) * x + r.random())).reshape(shape)
            f += amplitude * (0.5 + 0.5 * r.random()) * term
        return f

    drho = waves(0.2 * u_max)
    u = [waves(0.2 * u_max) for _ in range(dims)]  # x, y (, z)
    u[0] += 0.5 * u_max
    g = torch.zeros((len(c),) + cells.shape, device=dev, dtype=dtype)
    for i, ci in enumerate(c):
        cu = sum(k * v for k, v in zip(ci, u) if k)
        g[i] = torch.where(fluid, w[i] * (drho + 3.0 * cu), 0.0).to(dtype)
    return g


# ---- prepare, run, work --------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind, u_scale = case["kind"], 0.9 + 0.2 * random.Random(seed).random()
    if kind in ("advance2d", "loop2d"):
        cells = _cells(case)
        lat = L.Lattice(cells, case["tau"], _u_max(case, seed), precision=case["precision"],
                        collision=COLLISION[case["collision"]], c_smag=C_SMAG,
                        mirror=case["geometry"] == "collector")
        fields = {k: torch.zeros(cells.shape, device="cuda") for k in ("drho", "ux", "uy")}
        s = dict(case=case, lat=lat, fields=fields)
        if kind == "advance2d":
            s["state"] = _state(cells, seed, case["u_max"], STORAGE[case["precision"]])
            s["saved"] = torch.zeros_like(s["state"])
        else:
            s["mask"] = torch.zeros(cells.shape, dtype=torch.uint8, device="cuda")
            s["n_swap"] = max(1, _fluid(cells) // 500)
    elif kind in ("advance3d", "loop3d"):
        cells = _cells(case)
        lat = L.Lattice3(cells, case["tau"], _u_max(case, seed), precision=case["precision"],
                         collision=COLLISION[case["collision"]], c_smag=C_SMAG)
        fields = {k: torch.zeros(cells.shape, device="cuda") for k in ("drho", "ux", "uy", "uz")}
        state = _state(cells, seed, case["u_max"], STORAGE[case["precision"]])
        s = dict(case=case, lat=lat, fields=fields, state=state, saved=torch.zeros_like(state))
        if kind == "loop3d":
            s["mask"] = torch.zeros(cells.shape, dtype=torch.uint8, device="cuda")
            s["n_swap"] = max(1, _fluid(cells) // 500)
            s["cells"] = cells
            s["params"] = dict(tau=case["tau"], u_max=_u_max(case, seed), precision=case["precision"])
    elif kind == "batch":
        members = [dict(m, u_max=m["u_max"] * u_scale) for m in _candidates(case["n"], case["geo_seed"])]
        batch = L.Batch(members, precision=case["precision"])
        total = sum(m["cells"].size for m in members)
        s = dict(case=case, batch=batch, n_swap=[max(1, _fluid(m["cells"]) // 500) for m in members],
                 shapes=[m["cells"].shape for m in members],
                 mask=torch.zeros(total, dtype=torch.uint8, device="cuda"),
                 fields={k: torch.zeros(total, device="cuda") for k in ("drho", "ux", "uy")})
    else:
        reqs = [dict(r, u_max=r["u_max"] * u_scale, n_swap=max(1, _fluid(r["cells"]) // 500) if r["optimize"] else 0)
                for r in _requests(case["n"], case["geo_seed"])]
        s = dict(case=case, reqs=reqs, tags=itertools.count(),
                 server=L.Server(precision=case["precision"], max_active=1024, max_tick_steps=1000))
    torch.cuda.synchronize()
    return s


FIELDS2 = dict(drho=L.FIELD_DRHO, ux=L.FIELD_UX, uy=L.FIELD_UY)
FIELDS3 = dict(drho=L.FIELD3_DRHO, ux=L.FIELD3_UX, uy=L.FIELD3_UY, uz=L.FIELD3_UZ)


def _numbers(r, keys):
    return {k: r[k] for k in keys}


def run(state):
    s, case = state, state["case"]
    kind = case["kind"]
    if kind in ("advance2d", "advance3d"):
        two = kind == "advance2d"
        lat = s["lat"]
        lat.load_state(s["state"])
        r = lat.solve(case["steps"])
        for k, f in (FIELDS2 if two else FIELDS3).items():
            lat.read(f, out=s["fields"][k])
        lat.read(L.FIELD_POPS if two else L.FIELD3_POPS, out=s["saved"])
        keys = ("dp", "m_in", "m_out", "residual", "theta", "dg") if two else ("dp", "m_in", "m_out")
        return dict(_numbers(r, keys), saved=s["saved"], **s["fields"])
    if kind == "loop2d":
        lat = s["lat"]
        lat.reset()
        r = lat.optimize(case["steps"], case["iters"], s["n_swap"])
        for k, f in FIELDS2.items():
            lat.read(f, out=s["fields"][k])
        lat.read(L.FIELD_MASK, out=s["mask"])
        return dict(history=r["history"], swapped=r["swapped"], mask=s["mask"], **s["fields"])
    if kind == "loop3d":  # a 3D handle has no reset: every design starts on a handle of its own
        lat = L.Lattice3(s["cells"], s["params"]["tau"], s["params"]["u_max"], precision=s["params"]["precision"])
        lat.load_state(s["state"])
        r = lat.optimize(case["steps"], case["iters"], s["n_swap"])
        for k, f in FIELDS3.items():
            lat.read(f, out=s["fields"][k])
        lat.read(L.FIELD3_MASK, out=s["mask"])
        lat.close()
        return dict(history=r["history"], swapped=r["swapped"], mask=s["mask"], **s["fields"])
    if kind == "batch":
        b = s["batch"]
        b.reset()
        first = b.solve(case["steps"])
        then = b.optimize_step(s["n_swap"], case["steps"])
        at = 0
        for i, (ny, nx) in enumerate(s["shapes"]):
            b.read(i, L.FIELD_MASK, out=s["mask"][at:at + ny * nx])
            for k, f in FIELDS2.items():
                b.read(i, f, out=s["fields"][k][at:at + ny * nx])
            at += ny * nx
        return dict(dp_first=np.array([r["dp"] for r in first]), dp=np.array([r["dp"] for r in then]),
                    theta=np.array([r["theta"] for r in then]), m_out=np.concatenate([r["m_out"] for r in then]),
                    swapped=np.array([r["n_swapped"] for r in then]), mask=s["mask"], **s["fields"])
    # served: a client that optimises takes the shape and its flow, one that solves takes the numbers
    server = s["server"]
    tags = [next(s["tags"]) for _ in s["reqs"]]
    for t, r in zip(tags, s["reqs"]):
        server.submit(t, r["cells"], r["tau"], r["u_max"], case["steps"], n_iter=r["n_iter"], n_swap=r["n_swap"],
                      keep_fields=r["optimize"])
    done = {}
    while len(done) < len(tags):
        for d in server.poll(wait_ms=1000):
            done[d["tag"]] = d
    got = [done[t] for t in tags]
    shapes = [d["fields"] for d in got if "fields" in d]
    out = dict(status=np.array([d["status"] for d in got]), dp=np.array([d["last"]["dp"] for d in got]),
               dp_first=np.array([d["dp_first"] for d in got]),
               m_out=np.concatenate([d["last"]["m_out"] for d in got]),
               swapped=np.array([d["n_swapped"] for d in got]))
    for k in ("mask", "drho", "ux", "uy"):
        if shapes:
            out[k] = np.concatenate([f[k].reshape(-1) for f in shapes])
    return out


def work(case):
    """Of one pass: every solve reads and writes its fluid cells' populations once and writes their moments once
    (a solve's steps need not pass through memory), and updates them at every step."""
    kind = case["kind"]
    sb = 4 if case["precision"] == "f32" else 2
    if kind == "batch":
        fluid, updates = sum(_fluid(m["cells"]) for m in _candidates(case["n"], case["geo_seed"])), 0
        updates, solves = fluid * 2 * case["steps"], 2
    elif kind == "served":
        reqs = _requests(case["n"], case["geo_seed"])
        updates = sum(_fluid(r["cells"]) * case["steps"] * (1 + r["n_iter"]) for r in reqs)
        fluid, solves = updates // case["steps"], 1
    else:
        fluid = _fluid(_cells(case))
        solves = 1 + case.get("iters", 0)
        updates = fluid * solves * case["steps"]
    three = kind.endswith("3d")
    q, fields = (19, 4) if three else (9, 3)
    return {"bytes": solves * fluid * (2 * q * sb + 4 * fields), "flops": updates * (FLOPS3 if three else FLOPS2)}


# ---- the 64-bit statement ------------------------------------------------------------------------------------------

def exact(case, seed):
    """What an advance returns, in 64 bits: the fluid cells as one list, their incoming populations gathered from
    where they stream from (or from the cell's own reversed direction at a wall), the port rules, the collision.
    The other kinds exchange cells on the way, a choice among nearly equal scores that 64 bits need not share; the
    longest advances take too long."""
    if case["kind"].startswith("advance") and _fluid(_cells(case)) * case["steps"] > 4.5e9:
        return None
    if case["kind"] == "advance2d":
        return _exact(case, seed, C2, W2)
    if case["kind"] == "advance3d":
        return _exact(case, seed, C3, W3)
    return None


def _exact(case, seed, c, w):
    dims, q, dev = len(c[0]), len(c), "cuda"
    cells = _cells(case)
    shape = cells.shape
    f64 = dict(dtype=torch.float64, device=dev)
    solid = torch.from_numpy(cells).to(dev) != 0
    at = torch.nonzero(~solid.reshape(-1)).reshape(-1)
    n = at.numel()
    number = torch.full((solid.numel(),), -1, dtype=torch.int64, device=dev)
    number[at] = torch.arange(n, device=dev)
    nx, ny = shape[-1], shape[-2]
    x, rest = at % nx, at // nx
    y, z = rest % ny, rest // ny
    opp = [c.index(tuple(-k for k in ci)) for ci in c]
    src = torch.empty((q, n), dtype=torch.int64, device=dev)
    own = torch.arange(n, device=dev)
    for i, ci in enumerate(c):
        sx, sy, sz = x - ci[0], y - ci[1], z - (ci[2] if dims == 3 else 0)
        inside = (sx >= 0) & (sx < nx)  # rows outside the frame do not occur: the frame is solid
        k = number[(sz * ny + sy) * nx + sx.clamp(0, nx - 1)]
        src[i] = torch.where(inside & (k >= 0), i * n + k, opp[i] * n + own)
    start = _state(cells, seed, case["u_max"], STORAGE[case["precision"]])
    g = start.reshape(q, -1)[:, at].to(torch.float64)
    tau, u_max = case["tau"], _u_max(case, seed)
    omega = 1.0 / tau

    def run_of(a):  # of each True of a (..., n): its place s in its run along the last axis, 4 s (1 - s)
        out = np.zeros(a.shape)
        for idx in np.ndindex(a.shape[:-1]):
            row, k = a[idx], 0
            while k < row.size:
                if not row[k]:
                    k += 1
                    continue
                e = k
                while e < row.size and row[e]:
                    e += 1
                sp = (np.arange(e - k) + 0.5) / (e - k)
                out[idx][k:e] = 4 * sp * (1 - sp)
                k = e
        return out

    inlet, outlet = torch.nonzero(x == 0).reshape(-1), torch.nonzero(x == nx - 1).reshape(-1)
    port = cells[..., 0] == 0
    profile = run_of(port)
    if dims == 3:
        profile = profile * run_of(port.T).T
    u_in = torch.from_numpy(u_max * profile.reshape(-1)).to(dev)[rest[inlet]]
    cs = torch.tensor(c, **f64)
    ws = torch.tensor(w, **f64).reshape(q, 1)

    def equilibria(drho, u):
        rho = 1.0 + drho
        t0 = drho - 1.5 * rho * sum(v * v for v in u)
        e = torch.empty((q, drho.numel()), **f64)
        for i, ci in enumerate(c):
            cu = sum((v if k > 0 else -v) for k, v in zip(ci, u) if k)
            e[i] = w[i] * (t0 + 3 * rho * cu + 4.5 * rho * cu * cu) if any(ci) else w[i] * t0
        return e

    def stress(neq):
        return [[sum(ci[a] * ci[b] * neq[i] for i, ci in enumerate(c) if ci[a] * ci[b]) for b in range(dims)]
                for a in range(dims)]

    def projected(neq):  # w_i / (2 c_s^4) (c_i c_i - I / 3) : Pi
        p = stress(neq)
        tr = sum(p[a][a] for a in range(dims))
        return torch.stack([4.5 * w[i] * (sum(ci[a] * ci[b] * p[a][b] for a in range(dims) for b in range(dims))
                                          - tr / 3) for i, ci in enumerate(c)])

    def at_port(cellno, u, sign):
        gp = g_in[:, cellno]
        flat = gp[[i for i in range(q) if c[i][0] == 0]].sum(0)
        known = gp[[i for i in range(q) if c[i][0] == -sign]].sum(0)
        if sign > 0:
            drho, ux = (flat + 2 * known + u) / (1 - u), u
        else:
            ux = flat + 2 * known
            drho = torch.zeros_like(ux)
        e = equilibria(drho, [ux] + [torch.zeros_like(ux)] * (dims - 1))
        for i in range(q):
            if c[i][0] == sign:
                gp[i] = e[i] + (gp[opp[i]] - e[opp[i]])
        g_in[:, cellno] = e + projected(gp - e)

    steps, every = case["steps"], 100
    with_residual = dims == 2 and steps >= every + 2
    before = None
    for step in range(steps):
        g_in = g.reshape(-1)[src]
        at_port(inlet, u_in, 1)
        at_port(outlet, None, -1)
        drho = g_in.sum(0)
        rho = 1.0 + drho
        u = [sum((g_in[i] if ci[a] > 0 else -g_in[i]) for i, ci in enumerate(c) if ci[a]) / rho for a in range(dims)]
        e = equilibria(drho, u)
        if case["collision"] == "regularized":
            g = e + (1 - omega) * projected(g_in - e)
        elif case["collision"] == "smagorinsky":
            p = stress(g_in - e)
            pp = sum(p[a][b] ** 2 for a in range(dims) for b in range(dims))
            t = 0.5 * (tau + torch.sqrt(tau * tau + 18 * math.sqrt(2.0) * C_SMAG ** 2 * torch.sqrt(pp) / rho))
            g = g_in + (e - g_in) / t
        else:
            g = g_in + omega * (e - g_in)
        if with_residual and step == steps - 1 - every:
            before = u

    def spread(v, into=None):
        out = torch.zeros(solid.numel(), **f64) if into is None else into
        out[at] = v
        return out.reshape(shape)

    saved = start.reshape(q, -1).to(torch.float64)
    out = dict(drho=spread(drho))
    for k, v in zip(("ux", "uy", "uz"), u):
        out[k] = spread(v)
    out["saved"] = torch.stack([spread(g[i], saved[i]) for i in range(q)])
    out["dp"] = float((drho[inlet].mean() - drho[outlet].mean()) / 3)
    flow = rho * u[0]
    out["m_in"] = float(flow[inlet].sum())
    # outlets: the connected fluid regions of the last column, numbered from its first cell on
    open_ = cells[..., -1] == 0
    label = np.full(open_.shape, -1)
    count = 0
    for idx in zip(*np.nonzero(open_)):
        if label[idx] >= 0:
            continue
        stack, label[idx] = [idx], count
        while stack:
            k = stack.pop()
            for a in range(open_.ndim):
                for d in (-1, 1):
                    j = tuple(v + (d if b == a else 0) for b, v in enumerate(k))
                    if all(0 <= v < m for v, m in zip(j, open_.shape)) and open_[j] and label[j] < 0:
                        label[j] = count
                        stack.append(j)
        count += 1
    which = torch.from_numpy(label.reshape(-1)).to(dev)[rest[outlet]]
    m = torch.zeros(count, **f64).index_add_(0, which, flow[outlet]).cpu().numpy()
    out["m_out"] = m
    if dims == 2:
        out["theta"] = float(m.max() / m.min())
        out["dg"] = float(np.sqrt(np.sum((m / m.mean() - 1) ** 2) / (count - 1))) if count > 1 else 0.0
        if case["precision"] != "f32":  # ratios of outlet flows that may nearly vanish: 16-bit storage leaves them open
            out["m_out"] = out["theta"] = out["dg"] = None
        out["residual"] = -1.0
        if with_residual:
            du = sum((a - b).abs().sum() for a, b in zip(u, before))
            out["residual"] = float(du / sum(a.abs().sum() for a in u))
    return out
