"""Workloads of the library as user programs run them, for timing and for comparing results.

``listed()`` names twelve calls over the range of the public entry points (``paper_2209_13775_gb300.lcs``);
``draw(rng)`` gives more of the same ranges; ``prepare(case, seed)`` builds what a program holds before the
call (field, seed lattice, flow map, options, output buffers); ``run(state)`` is one pass; ``work(case)`` is
the least traffic and arithmetic of a pass; ``exact(case, seed)`` is the same pass in plain FP64 torch.

A program keeps one context per host thread, so the module keeps one context per process.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2209_13775_gb300 import inputs, lcs

DEV = "cuda"
GYRE_BOX = (2.0, 1.0)
TWO_PI = 2.0 * math.pi
DUCT_LENGTH = 10.0
STORAGE = {"f32": lcs.F32, "f16": lcs.F16, "bf16": lcs.BF16}
STORE_DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
EXACT_MOST_2D, EXACT_MOST_3D, EXACT_MOST_MESH = 4.0e9, 8.0e8, 2.5e9   # tracer-steps integrated in FP64


def listed():
    return [
        # one interactive FTLE of a coarse lattice: launches and host calls are what counts
        {"name": "gyre_small", "path": "gyre", "nx": 64, "ny": 32, "jobs": 1, "t_long": 5.0, "storage": "f32"},
        # sliding-window FTLE: 64 windows, both directions, on a 2048 x 1024 lattice (graph replayed each pass)
        {"name": "gyre_windows", "path": "gyre", "nx": 2048, "ny": 1024, "jobs": 64, "t_long": 8.0, "storage": "f32"},
        # one adaptive DP5(4) integration of the 2D lattice
        {"name": "gyre_rk45", "path": "gyre_rk45", "nx": 1024, "ny": 512, "t_long": 8.0, "storage": "f32"},
        # the 3D workload: 256^3 seeds, 400 steps, FTLE with the Cauchy-Green tensor written
        {"name": "abc_lattice", "path": "abc", "grid": 128, "nframes": 64, "side": 256, "steps": 400,
         "storage": "f32"},
        # 3D data arriving frame block by frame block in reduced precision, on a small ragged lattice
        {"name": "abc_stream_f16", "path": "abc_stream", "grid": 64, "nframes": 16, "side": 47, "steps": 100,
         "storage": "f16"},
        # grad F by the variational equations next to the 3D trajectories
        {"name": "abc_variational", "path": "abc_var", "grid": 128, "nframes": 16, "side": 128, "steps": 100,
         "storage": "f32"},
        # adaptive DP5(4) through a tetrahedral mesh of about a million cells
        {"name": "duct_rk45", "path": "duct_rk45", "m": 16, "nx": 64, "nz": 512, "storage": "f32"},
        # fixed-step RK4 through a tetrahedral mesh, velocity kept in BF16, odd lattice
        {"name": "duct_rk4_bf16", "path": "duct_rk4", "m": 12, "nx": 45, "nz": 301, "steps": 100, "storage": "bf16"},
        # fixed-step RK4 through a triangle mesh of 1.6 million cells
        {"name": "stenosis_rk4", "path": "stenosis", "h": 0.005, "nx": 4096, "ny": 1024, "steps": 500,
         "storage": "f32"},
        # the surrogate network evaluated at every point of a lattice (ragged count)
        {"name": "network", "path": "network", "n": 2097152 + 77},
        # one optimiser step of the surrogate network on a batch of 65,536 samples
        {"name": "train_step", "path": "train", "n": 65536},
        # all eigenpairs of C at every seed
        {"name": "abc_eigen", "path": "abc_eigen", "grid": 64, "nframes": 8, "side": 160, "steps": 100,
         "storage": "f32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["gyre", "gyre", "gyre_rk45", "abc", "abc", "abc_stream", "abc_var", "duct_rk45", "duct_rk4",
                       "stenosis", "network", "train", "abc_eigen"])
    st = rng.choice(["f32", "f32", "f16", "bf16"])
    if path == "gyre":
        nx = _log(rng, 24, 2048)
        return {"path": path, "nx": nx, "ny": max(9, nx // 2 - rng.randrange(0, 4)),
                "jobs": _log(rng, 1, 64), "t_long": 0.05 * rng.randrange(20, 161), "storage": st}
    if path == "gyre_rk45":
        nx = _log(rng, 64, 2048)
        return {"path": path, "nx": nx, "ny": nx // 2 - rng.randrange(0, 4), "t_long": rng.uniform(2.0, 10.0),
                "storage": st}
    if path == "abc":
        return {"path": path, "grid": rng.randrange(48, 129), "nframes": rng.randrange(8, 65),
                "side": _log(rng, 24, 256), "steps": rng.randrange(20, 401), "storage": st}
    if path == "abc_stream":
        return {"path": path, "grid": rng.randrange(32, 97), "nframes": rng.randrange(2, 25),
                "side": _log(rng, 17, 96), "steps": rng.randrange(20, 201), "storage": st}
    if path == "abc_var":
        return {"path": path, "grid": rng.randrange(48, 129), "nframes": rng.randrange(4, 25),
                "side": _log(rng, 24, 160), "steps": rng.randrange(20, 161), "storage": st}
    if path in ("duct_rk45", "duct_rk4"):
        c = {"path": path, "m": rng.randrange(6, 17), "nx": rng.randrange(15, 65), "nz": _log(rng, 33, 512),
             "storage": st}
        if path == "duct_rk4":
            c["steps"] = rng.randrange(20, 101)
        return c
    if path == "stenosis":
        nx = _log(rng, 128, 4096)
        return {"path": path, "h": rng.choice([0.005, 0.01, 0.02, 0.04]), "nx": nx,
                "ny": nx // 4 - rng.randrange(0, 4), "steps": rng.randrange(50, 501), "storage": st}
    if path == "network":
        return {"path": path, "n": _log(rng, 1000, 4000000)}
    if path == "train":
        return {"path": path, "n": 128 * _log(rng, 8, 1024)}
    return {"path": "abc_eigen", "grid": rng.randrange(32, 97), "nframes": rng.randrange(4, 17),
            "side": _log(rng, 24, 224), "steps": rng.randrange(20, 101), "storage": st}


# ------------------------------------------------------------------ inputs

def _uniform(seed, n):
    """n numbers in [0, 1) of the seed."""
    return np.random.default_rng(seed).random(n)


def _gyre_field(case, seed):
    """Double gyre, 129 x 65 nodes, 101 frames of one period, amplitude and phase of the seed (FP32, device)."""
    r = _uniform(seed, 3)
    amp, eps, ph = 0.08 + 0.04 * r[0], 0.2 + 0.1 * r[1], TWO_PI * r[2]
    nx, ny, nf, omega = 129, 65, 101, TWO_PI / 10.0
    x = torch.linspace(0.0, 2.0, nx, dtype=torch.float64, device=DEV)
    y = torch.linspace(0.0, 1.0, ny, dtype=torch.float64, device=DEV)[:, None]
    times = np.array([10.0 * k / (nf - 1) for k in range(nf)])
    frames = torch.empty((nf, ny, nx, 2), dtype=torch.float32, device=DEV)
    for k, t in enumerate(times):
        a = eps * math.sin(omega * t + ph)
        b = 1.0 - 2.0 * a
        f, df = math.pi * (a * x * x + b * x), 2.0 * a * x + b
        frames[k, :, :, 0] = -math.pi * amp * torch.sin(f) * torch.cos(math.pi * y)
        frames[k, :, :, 1] = math.pi * amp * torch.cos(f) * torch.sin(math.pi * y) * df
    geom = {"dim": 2, "n": (nx, ny), "origin": (0.0, 0.0), "spacing": (2.0 / (nx - 1), 1.0 / (ny - 1)),
            "periodic": (0, 0), "times": times, "time_periodic": True, "period": 10.0}
    return frames, geom


def _abc_field(case, seed):
    """Time-modulated ABC flow on a periodic grid, coefficients and phases of the seed (FP32, device)."""
    n, nf = case["grid"], case["nframes"]
    r = _uniform(seed, 6)
    A, B, C = math.sqrt(3.0) * (0.95 + 0.1 * r[0]), math.sqrt(2.0) * (0.95 + 0.1 * r[1]), 0.95 + 0.1 * r[2]
    h, t_end = TWO_PI / n, max(8.0 * nf / 64.0, 0.02 * case["steps"])
    g = torch.arange(n, dtype=torch.float64, device=DEV) * h
    x, y, z = (g + TWO_PI * r[3])[None, None, :], (g + TWO_PI * r[4])[None, :, None], (g + TWO_PI * r[5])[:, None, None]
    times = np.array([t_end * k / max(nf - 1, 1) for k in range(nf)])
    frames = torch.empty((nf, n, n, n, 3), dtype=torch.float32, device=DEV)
    for k, t in enumerate(times):
        At = A + 0.5 * t * math.sin(math.pi * t)
        frames[k, ..., 0] = At * torch.sin(z) + C * torch.cos(y)
        frames[k, ..., 1] = B * torch.sin(x) + At * torch.cos(z)
        frames[k, ..., 2] = C * torch.sin(y) + B * torch.cos(x)
    geom = {"dim": 3, "n": (n, n, n), "origin": (0.0,) * 3, "spacing": (h, h, h), "periodic": (1, 1, 1),
            "times": times, "time_periodic": False, "period": 0.0}
    return frames, geom


@functools.lru_cache(maxsize=2)
def _duct_mesh(m):
    """Box [-1, 1]^2 x [0, 10] of cubes of side 1/m, six tets around each cube's diagonal, interior nodes moved
    by up to a tenth of a cube (nodes FP32 [nn][3], tets and face neighbours int32 [nc][4])."""
    nx, nz = 2 * m, int(DUCT_LENGTH) * m
    ax, az = np.arange(nx + 1), np.arange(nz + 1)
    K, J, I = np.meshgrid(az, ax, ax, indexing="ij")
    P = np.stack([I, J, K], -1).reshape(-1, 3).astype(np.float64)
    hi = np.array([nx, nx, nz])
    inner = ((P > 0) & (P < hi)).all(axis=1)
    P[inner] += np.random.default_rng(7).uniform(-0.1, 0.1, (int(inner.sum()), 3))
    xyz = (P / m - np.array([1.0, 1.0, 0.0])).astype(np.float32)
    k, j, i = (a.ravel() for a in np.meshgrid(az[:-1], ax[:-1], ax[:-1], indexing="ij"))
    step = (1, nx + 1, (nx + 1) ** 2)
    base = i + (nx + 1) * (j + (nx + 1) * k)
    tets = np.empty((base.size, 6, 4), dtype=np.int64)
    for q, perm in enumerate([(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]):
        v = base
        tets[:, q, 0] = v
        for a, axis in enumerate(perm):
            v = v + step[axis]
            tets[:, q, a + 1] = v
    tets = tets.reshape(-1, 4)
    t = torch.from_numpy(tets).to(DEV)
    faces = torch.stack([t[:, [1, 2, 3]], t[:, [0, 2, 3]], t[:, [0, 1, 3]], t[:, [0, 1, 2]]], 1).reshape(-1, 3)
    faces = faces.sort(dim=1).values
    nn = xyz.shape[0]
    key, order = ((faces[:, 0] * nn + faces[:, 1]) * nn + faces[:, 2]).sort()
    pair = torch.nonzero(key[1:] == key[:-1]).ravel()
    nbrs = torch.full((faces.shape[0],), -1, dtype=torch.int64, device=DEV)
    nbrs[order[pair]] = order[pair + 1] // 4
    nbrs[order[pair + 1]] = order[pair] // 4
    return xyz, tets.astype(np.int32), nbrs.reshape(-1, 4).to(torch.int32).cpu().numpy()


def _duct_field(case, seed):
    """Pulsatile flow along the duct plus a swirl that vanishes on its walls (FP32, device; 51 frames of a period)."""
    mesh = _duct_mesh(case["m"])
    r = _uniform(seed, 5)
    p = torch.from_numpy(mesh[0]).to(DEV, torch.float64)
    wall = (1.0 - p[:, 0] ** 2) * (1.0 - p[:, 1] ** 2)
    times = np.array([k / 50.0 for k in range(51)])
    frames = torch.empty((51, p.shape[0], 3), dtype=torch.float32, device=DEV)
    for k, t in enumerate(times):
        sw = sum(torch.sin(TWO_PI * (q * p[:, 2] / DUCT_LENGTH + r[q - 1] + t)) / q for q in range(1, 5))
        frames[k, :, 0] = -0.15 * wall * sw * p[:, 1]
        frames[k, :, 1] = 0.15 * wall * sw * p[:, 0]
        frames[k, :, 2] = wall * (1.0 + 0.5 * math.sin(TWO_PI * (t + r[4])))
    return frames, {"dim": 3, "kind": lcs.TET, "mesh": mesh, "times": times, "time_periodic": True, "period": 1.0}


@functools.lru_cache(maxsize=2)
def _stenosis_mesh(h):
    mesh = inputs.stenosis_mesh(h=h)
    return mesh.xyz, mesh.tets, mesh.nbrs, mesh.extra


def _halfwidth(x, ex):
    e = torch.exp(-((x - ex["xc"]) / ex["w"]) ** 2)
    return ex["H"] * (1.0 - ex["depth"] * e), 2.0 * ex["H"] * ex["depth"] * e * (x - ex["xc"]) / ex["w"] ** 2


def _stenosis_field(case, seed):
    """Pulsatile channel flow through a constriction with a travelling wave (FP32, device; 41 frames of a period)."""
    xy, tris, nbrs, ex = _stenosis_mesh(case["h"])
    r = _uniform(seed, 2)
    p = torch.from_numpy(xy).to(DEV, torch.float64)
    x, y = p[:, 0], p[:, 1]
    hw, dhw = _halfwidth(x, ex)
    s = y / hw
    ds = -s * dhw / hw
    fp, g, gp = 1.5 * (1.0 - s * s), (1.0 - s * s) ** 2, -4.0 * s * (1.0 - s * s)
    times = np.array([k / 40.0 for k in range(41)])
    frames = torch.empty((41, x.numel(), 2), dtype=torch.float32, device=DEV)
    for q, t in enumerate(times):
        Q = 1.0 + 0.5 * math.sin(TWO_PI * (t + r[0]))
        ph = math.pi * (x - 2.0 * t) + TWO_PI * r[1]
        frames[q, :, 0] = Q * fp / hw + 0.05 * gp * torch.sin(ph) / hw
        frames[q, :, 1] = -(Q * fp * ds + 0.05 * (gp * ds * torch.sin(ph) + g * math.pi * torch.cos(ph)))
    return frames, {"dim": 2, "kind": lcs.TRI, "mesh": (xy, tris, nbrs), "extra": ex, "times": times,
                    "time_periodic": True, "period": 1.0}


def _jobs(case):
    """Start times and horizons of the sliding windows: half forward, half backward, long, half and quarter ones."""
    nj, long = case["jobs"], int(round(case["t_long"] / 0.05))
    T = [0.05 * max(1, long // (1, 2, 4)[j % 3]) * (1 if j % 2 == 0 else -1) for j in range(nj)]
    return [0.25 * (j // 2) for j in range(nj)], T


FIELDS = {"gyre": _gyre_field, "gyre_rk45": _gyre_field, "abc": _abc_field, "abc_stream": _abc_field,
          "abc_var": _abc_field, "abc_eigen": _abc_field, "duct_rk45": _duct_field, "duct_rk4": _duct_field,
          "stenosis": _stenosis_field}


def _lattice(case):
    """(n, lo, hi, periodic) of the case's seed lattice."""
    p = case["path"]
    if p.startswith("gyre"):
        return (case["nx"], case["ny"]), (0.0, 0.0), GYRE_BOX, (0, 0)
    if p.startswith("abc"):
        s = case["side"]
        n = (s, s + 2, s - 2) if p == "abc_stream" else (s, s, s)
        return n, (0.0,) * 3, (TWO_PI,) * 3, (1, 1, 1)
    if p.startswith("duct"):
        return (case["nx"], case["nx"], case["nz"]), (-0.95, -0.95, 0.05), (0.95, 0.95, 9.95), (0, 0, 0)
    return (case["nx"], case["ny"]), (0.0, -1.0), (10.0, 1.0), (0, 0)


MLP = {"center": (1.0, 0.5), "kx": math.pi, "ky": math.pi, "omega": TWO_PI / 10.0, "tau": 0.5, "out_scale": 0.1}
RHO_WEIGHT, LR = 0.01, 1e-3


def _points(n, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    u = torch.rand((3, n), generator=g, device=DEV, dtype=torch.float32)
    return u * torch.tensor([[2.0], [1.0], [10.0]], device=DEV)


def _displacements(xyt, seed):
    """Smooth displacements over one network step with the size the gyre gives them."""
    a = TWO_PI * float(_uniform(seed, 1)[0])
    x, y, t = xyt[0], xyt[1], xyt[2]
    s = 0.1 * torch.sin(TWO_PI * t / 10.0 + a)
    return torch.stack([-0.15 * torch.sin(math.pi * (x + s)) * torch.cos(math.pi * y),
                        0.15 * torch.cos(math.pi * (x + s)) * torch.sin(math.pi * y)]).contiguous()


# ------------------------------------------------------------------- state

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = lcs.lcs_create(torch.cuda.current_device(), torch.cuda.current_stream())
    return _ctx


class State:
    """The handles and buffers of one case; the handles are freed with it."""

    def __init__(self, case):
        self.case, self.ctx, self.free = case, _context(), []

    def own(self, handle, free):
        self.free.append((free, handle))
        return handle

    def __del__(self):
        for free, handle in reversed(self.free):
            free(handle)


def prepare(case, seed):
    s = State(case)
    path = case["path"]
    if path in ("network", "train"):
        n = case["n"]
        s.params = torch.from_numpy(inputs.mlp_init(seed=seed)).to(DEV)
        s.mlp = s.own(lcs.lcs_mlp_create(s.ctx, lcs.mlp_desc(**MLP), s.params), lcs.lcs_mlp_free)
        s.xyt = _points(n, seed)
        if path == "network":
            s.out = torch.empty((3, n), device=DEV)
        else:
            s.disp = _displacements(s.xyt, seed)
            s.grads = torch.empty(lcs.MLP_NPARAMS, device=DEV)
        return s
    frames, g = FIELDS[path](case, seed)
    desc = lcs.field_desc(g["dim"], n=g.get("n", (1, 1, 1)), origin=g.get("origin", (0, 0, 0)),
                          spacing=g.get("spacing", (1, 1, 1)), periodic=g.get("periodic", (0, 0, 0)),
                          times=g["times"], time_periodic=g["time_periodic"], period=g["period"],
                          storage=STORAGE[case["storage"]], kind=g.get("kind", lcs.RECTILINEAR), mesh=g.get("mesh"))
    s.field = s.own(lcs.lcs_load_field(s.ctx, desc, frames), lcs.lcs_free_field)
    if path == "abc_stream":
        s.frames = frames
    n, lo, hi, per = _lattice(case)
    s.seeds = s.own(lcs.lcs_seed_grid(s.ctx, lcs.seed_desc(g["dim"], n, lo, hi, per), s.field), lcs.lcs_free_seeds)
    N, dim = lcs.lcs_seeds_count(s.seeds), g["dim"]
    nj = case.get("jobs", 1)
    s.fm = s.own(lcs.lcs_flowmap_create(s.ctx, s.seeds, nj), lcs.lcs_free_flowmap)
    s.ftle = torch.empty((nj, N), device=DEV)
    if path == "gyre":
        t0, T = _jobs(case)
        # one window is a plain call; a batch keeps the launch plan that the autotuner picks for it
        plan = {"variant": 5, "use_graph": True} if nj > 1 else {}
        s.opts = lcs.advect_opts(lcs.RK4, dt=0.05, job_t0=t0, job_T=T, **plan)
    elif path == "gyre_rk45":
        s.opts = lcs.advect_opts(lcs.RK45, t0=0.0, T=case["t_long"], rtol=1e-6, atol=1e-6, h0=0.05)
        s.xyz = torch.empty((dim, N), device=DEV)
    elif path.startswith("abc"):
        s.opts = lcs.advect_opts(lcs.RK4, t0=0.0, T=0.02 * case["steps"], dt=0.02, variational=path == "abc_var")
        if path in ("abc", "abc_stream"):
            s.C = torch.empty((N, 6), dtype=torch.float64, device=DEV)
        elif path == "abc_var":
            s.grad = torch.empty((N, 3, 3), device=DEV)
        else:
            s.eigval = torch.empty((N, 3), dtype=torch.float64, device=DEV)
            s.eigvec = torch.empty((N, 3, 3), dtype=torch.float64, device=DEV)
            lcs.lcs_advect(s.ctx, s.field, s.seeds, s.opts, s.fm)
    else:
        if path == "duct_rk45":
            s.opts = lcs.advect_opts(lcs.RK45, t0=0.0, T=1.0, rtol=1e-6, atol=1e-6, h0=0.02)
        elif path == "duct_rk4":
            s.opts = lcs.advect_opts(lcs.RK4, t0=0.0, T=0.01 * case["steps"], dt=0.01)
        else:
            s.opts = lcs.advect_opts(lcs.RK4, t0=0.0, T=0.002 * case["steps"], dt=0.002)
        s.xyz = torch.empty((dim, N), device=DEV)
        s.status = torch.empty(N, dtype=torch.uint8, device=DEV)
    return s


def run(s):
    path, ctx = s.case["path"], s.ctx
    if path == "network":
        lcs.lcs_mlp_forward(ctx, s.mlp, s.xyt, s.out)
        return {"out": s.out}
    if path == "train":
        loss = lcs.lcs_mlp_loss_grad(ctx, s.mlp, s.xyt, s.disp, RHO_WEIGHT, s.grads)
        lcs.lcs_mlp_adam(ctx, s.mlp, lr=LR)
        lcs.lcs_mlp_get_params(ctx, s.mlp, s.params)
        return {"loss": loss, "grads": s.grads, "params": s.params}
    if path == "abc_eigen":
        lcs.lcs_cg_eigen(ctx, s.fm, 0, s.eigval, s.eigvec)
        return {"eigval": s.eigval, "eigvec": s.eigvec}
    if path == "abc_stream":
        lcs.lcs_update_frames(ctx, s.field, s.frames)
    lcs.lcs_advect(ctx, s.field, s.seeds, s.opts, s.fm)
    if path == "gyre":
        lcs.lcs_ftle(ctx, s.fm, -1, s.ftle)
        return {"ftle": s.ftle}
    if path == "abc_var":
        lcs.lcs_ftle_variational(ctx, s.fm, 0, s.ftle)
        lcs.lcs_flowmap_grad(ctx, s.fm, 0, s.grad)
        return {"ftle": s.ftle, "grad": s.grad}
    if path.startswith("abc"):
        lcs.lcs_ftle(ctx, s.fm, 0, s.ftle, None, s.C)
        return {"ftle": s.ftle, "C": s.C}
    lcs.lcs_ftle(ctx, s.fm, 0, s.ftle)
    if path == "gyre_rk45":
        lcs.lcs_flowmap_get(ctx, s.fm, 0, s.xyz)
        return {"ftle": s.ftle, "xyz": s.xyz}
    lcs.lcs_flowmap_get(ctx, s.fm, 0, s.xyz, s.status)
    return {"ftle": s.ftle, "xyz": s.xyz, "status": s.status}


def work(case):
    """Fields, seeds and outputs moved once; arithmetic of the stage evaluations, differences and eigenvalues."""
    path = case["path"]
    if path == "network":
        return {"bytes": 24.0 * case["n"], "flops": 100864.0 * case["n"]}
    if path == "train":
        return {"bytes": 20.0 * case["n"] + 4.0 * lcs.MLP_NPARAMS * 8, "flops": 3.0 * 100864.0 * case["n"]}
    n = _lattice(case)[0]
    N, dim = math.prod(n), len(n)
    item = 4 if case["storage"] == "f32" else 2
    if path.startswith("gyre"):
        nodes, nf = 129 * 65, 101
    elif path.startswith("abc"):
        nodes, nf = case["grid"] ** 3, case["nframes"]
    elif path.startswith("duct"):
        nodes, nf = (2 * case["m"] + 1) ** 2 * (10 * case["m"] + 1), 51
    else:
        nodes, nf = int(10 / case["h"] + 1) * int(2 / case["h"] + 1), 41
    field, nj = float(nodes * nf * dim * item), 1
    cg = 40.0 if dim == 2 else 120.0
    if path == "abc_eigen":
        return {"bytes": N * (12.0 + 1 + 96), "flops": 400.0 * N}
    if path == "gyre":
        T = _jobs(case)[1]
        nj, steps, per = len(T), sum(int(round(abs(t) / 0.05)) for t in T), 164.0
    elif path == "gyre_rk45":
        steps, per = 4.0 * case["t_long"], 300.0
    elif path == "duct_rk45":
        steps, per = 10.0, 700.0
    else:
        steps = case["steps"]
        per = {"abc_var": 870.0, "duct_rk4": 400.0, "stenosis": 190.0}.get(path, 440.0)
    out = 4.0 + {"abc": 48.0, "abc_stream": 48.0, "abc_var": 36.0, "gyre": 0.0}.get(path, 4.0 * dim + 1)
    if path == "abc_stream":
        field = 4.0 * nodes * nf * dim
    return {"bytes": field + 4.0 * dim * N + out * N * nj, "flops": float(N) * (steps * per + nj * cg)}


# ---------------------------------------------- the same passes in FP64 torch

def _bracket(times, t, tp, period):
    """Frame k and the weight of frame k + 1 at time t."""
    if len(times) < 2:
        return 0, 0.0
    if tp:
        t = t - period * math.floor((t - times[0]) / period)
    k = min(max(int(np.searchsorted(times, t, side="right")) - 1, 0), len(times) - 2)
    a = (t - times[k]) / (times[k + 1] - times[k])
    return k, a if tp else min(max(a, 0.0), 1.0)


class _Rect:
    """Bilinear / trilinear interpolation in space (x [dim][N]), linear in time."""

    def __init__(self, frames, g, storage):
        self.g, self.dim = g, g["dim"]
        self.F = frames.to(STORE_DTYPE[storage]).reshape(frames.shape[0], -1, self.dim)

    def blend(self, t):
        k, a = _bracket(self.g["times"], t, self.g["time_periodic"], self.g["period"])
        u = self.F[k].double()
        return u if a == 0.0 else (1.0 - a) * u + a * self.F[k + 1].double()

    def corners(self, x):
        """Node ids and fractions: per axis ((i0, i1), f, moves)."""
        out = []
        for d in range(self.dim):
            n, h, o = self.g["n"][d], self.g["spacing"][d], self.g["origin"][d]
            s = (x[d] - o) / h
            if self.g["periodic"][d]:
                i = torch.floor(s)
                f = s - i
                i = i.long() % n
                out.append((i, (i + 1) % n, f, torch.ones_like(f, dtype=torch.bool)))
            else:
                on = (s >= 0) & (s <= n - 1)
                s = s.clamp(0, n - 1)
                i = s.long().clamp(max=n - 2)
                out.append((i, i + 1, s - i, on))
        return out

    def eval(self, x, u, grad=False):
        ax = self.corners(x)
        n = self.g["n"]
        val = torch.zeros((x.shape[1], self.dim), dtype=torch.float64, device=x.device)
        J = torch.zeros((x.shape[1], self.dim, self.dim), dtype=torch.float64, device=x.device) if grad else None
        for q in range(1 << self.dim):
            v, w, stride = 0, 1.0, 1
            bits = [(q >> d) & 1 for d in range(self.dim)]
            for d in range(self.dim):
                v = v + ax[d][bits[d]] * stride
                stride *= n[d]
            fs = [ax[d][2] if bits[d] else 1.0 - ax[d][2] for d in range(self.dim)]
            uq = u[v]
            val += math.prod(fs[1:], start=fs[0])[:, None] * uq
            if grad:
                for d in range(self.dim):
                    w = math.prod((fs[e] for e in range(self.dim) if e != d),
                                  start=(1.0 if bits[d] else -1.0) / self.g["spacing"][d] * ax[d][3].double())
                    J[:, :, d] += w[:, None] * uq
        return val.T, J

    def at(self, x, k, a):
        """u at x [dim][N] with a frame and weight per point."""
        nodes = self.F.shape[1]
        F = self.F.reshape(-1, self.dim)
        ax, val, ok = self.corners(x), 0.0, torch.ones(x.shape[1], dtype=torch.bool, device=x.device)
        for q in range(1 << self.dim):
            v, w, stride = 0, 1.0, 1
            for d in range(self.dim):
                b = (q >> d) & 1
                v = v + ax[d][b] * stride
                w = w * (ax[d][2] if b else 1.0 - ax[d][2])
                stride *= self.g["n"][d]
            v = v + k * nodes
            val = val + w[:, None] * ((1.0 - a)[:, None] * F[v].double() + a[:, None] * F[v + nodes].double())
        return val.T, ok

    def left(self, x):
        out = torch.zeros(x.shape[1], dtype=torch.bool, device=x.device)
        for d in range(self.dim):
            if not self.g["periodic"][d]:
                n, h, o = self.g["n"][d], self.g["spacing"][d], self.g["origin"][d]
                out |= (x[d] < o - h) | (x[d] > o + n * h)
        return out


class _Mesh:
    """P1 interpolation on tets or triangles: a walk in FP64 from the cell of the last point."""

    def __init__(self, frames, g, storage):
        self.g, self.dim = g, g["dim"]
        self.F = frames.to(STORE_DTYPE[storage])
        xyz, cells, nbrs = (torch.from_numpy(a).to(DEV) for a in g["mesh"])
        self.cells, self.nbrs = cells.long(), nbrs.long()
        p = xyz.double()[self.cells]
        self.v0 = p[:, 0]
        self.M = torch.linalg.inv((p[:, 1:] - p[:, :1]).transpose(1, 2))

    def bary(self, c, x):
        lam = torch.einsum("nij,jn->ni", self.M[c], x - self.v0[c].T)
        return torch.cat([1.0 - lam.sum(1, keepdim=True), lam], 1)

    def locate(self, x, cell):
        """(cell, inside) of every point; cell holds where to start."""
        cell, inside = cell.clone(), torch.zeros(x.shape[1], dtype=torch.bool, device=x.device)
        todo, edge = torch.arange(x.shape[1], device=x.device), []
        for _ in range(4096):
            if todo.numel() == 0:
                break
            lam = self.bary(cell[todo], x[:, todo])
            low, j = lam.min(dim=1)
            done = low >= -1e-6
            inside[todo[done]] = True
            nxt = self.nbrs[cell[todo], j]
            go = ~done & (nxt >= 0)
            edge.append(todo[~done & (nxt < 0)])
            cell[todo[go]] = nxt[go]
            todo = todo[go]
        if self.dim == 2:   # the channel is not convex: try every triangle for points the walk lost inside its box
            e = torch.cat(edge)
            e = e[(x[0, e] >= 0.0) & (x[0, e] <= 10.0)]
            e = e[x[1, e].abs() <= _halfwidth(x[0, e], self.g["extra"])[0] * (1 + 1e-3)]
            for q in e.tolist():
                d = x[:, q] - self.v0
                lam = torch.einsum("nij,nj->ni", self.M, d)
                hit = torch.nonzero(torch.minimum(lam.min(1).values, 1.0 - lam.sum(1)) >= -1e-6).ravel()
                if hit.numel():
                    cell[q], inside[q] = hit[0], True
        return cell, inside

    def p1(self, x, cell, u):
        return torch.einsum("ni,nid->dn", self.bary(cell, x), u[self.cells[cell]])


def _lattice_points(case):
    n, lo, hi, per = _lattice(case)
    axes = []
    for d in range(len(n)):
        step = (hi[d] - lo[d]) / (n[d] if per[d] else n[d] - 1)
        axes.append(torch.from_numpy((lo[d] + np.arange(n[d]) * step).astype(np.float32)).to(DEV, torch.float64))
    grid = torch.meshgrid(*axes[::-1], indexing="ij")[::-1]
    return torch.stack([a.reshape(-1) for a in grid])


def _rk4_rect(F, x, t0, T, dt, M=None):
    """x(t0 + T), status (0 in the domain, 1 left) and, with M, the variational grad F."""
    h = math.copysign(dt, T)
    x = x.clone()
    status = torch.zeros(x.shape[1], dtype=torch.uint8, device=x.device)
    c = (0.0, 0.5 * h, 0.5 * h, h)
    for n in range(int(round(abs(T) / dt))):
        t = t0 + n * h
        at = [F.blend(t), F.blend(t + 0.5 * h), F.blend(t + h)]
        k, K = [], []
        for s in range(4):
            y = x if s == 0 else x + c[s] * k[-1]
            v, J = F.eval(y, at[(0, 1, 1, 2)[s]], M is not None)
            k.append(v)
            if M is not None:
                K.append(J @ (M if s == 0 else M + c[s] * K[-1]))
        xn = x + h / 6.0 * (k[0] + 2.0 * k[1] + 2.0 * k[2] + k[3])
        x = torch.where(status == 0, xn, x)
        if M is not None:
            M = M + h / 6.0 * (K[0] + 2.0 * K[1] + 2.0 * K[2] + K[3])
        if not all(F.g["periodic"]):
            status[(status == 0) & F.left(x)] = 1
    return x, status, M


def _rk4_mesh(F, x, cell, status, T, dt):
    x = x.clone()
    for n in range(int(round(T / dt))):
        live = torch.nonzero(status == 0).ravel()
        y0, cl = x[:, live], cell[live]
        ok = torch.ones(live.numel(), dtype=torch.bool, device=x.device)
        k = []
        for s in range(4):
            y = y0 if s == 0 else y0 + (0.0, 0.5 * dt, 0.5 * dt, dt)[s] * k[-1]
            cl, inside = F.locate(y, cl)
            ok &= inside
            kk, a = _bracket(F.g["times"], n * dt + (0.0, 0.5, 0.5, 1.0)[s] * dt, True, F.g["period"])
            k.append(F.p1(y, cl, (1.0 - a) * F.F[kk].double() + a * F.F[kk + 1].double()))
        x[:, live] = torch.where(ok, y0 + dt / 6.0 * (k[0] + 2.0 * k[1] + 2.0 * k[2] + k[3]), y0)
        cell[live] = cl
        status[live[~ok]] = 1
    return x, status


DP_C = (0.0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1.0, 1.0)
DP_A = ((), (1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
        (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
        (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
        (35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
DP_E = (35 / 384 - 5179 / 57600, 0.0, 500 / 1113 - 7571 / 16695, 125 / 192 - 393 / 640, -2187 / 6784 + 92097 / 339200,
        11 / 84 - 187 / 2100, -1 / 40)


def _rk45(evaluate, left, x, status, T, h0, tol=1e-6):
    """Dormand-Prince 5(4) with one step size per 32 consecutive seeds; evaluate(points, ids, k, a) -> (u, inside)."""
    N = x.shape[1]
    G = (N + 31) // 32
    x = x.clone()
    group = torch.arange(N, device=x.device) // 32
    t, h = (torch.full((G,), v, dtype=torch.float64, device=x.device) for v in (0.0, h0))
    for _ in range(4000):
        live_g = torch.zeros(G, dtype=torch.bool, device=x.device)
        live_g[group[status == 0]] = True
        live_g &= t < T
        ids = torch.nonzero((status == 0) & live_g[group]).ravel()
        if ids.numel() == 0:
            break
        gi = group[ids]
        last = t + h >= T
        hs = torch.where(last, T - t, h)
        y0, hh, tt = x[:, ids], hs[gi], t[gi]
        ok = torch.ones(ids.numel(), dtype=torch.bool, device=x.device)
        k = []
        for s in range(7):
            y = y0 + hh * sum(a * v for a, v in zip(DP_A[s], k)) if s else y0
            u, inside = evaluate(y, ids, tt + DP_C[s] * hh)
            ok &= inside
            k.append(u)
        xn = y0 + hh * sum(a * v for a, v in zip(DP_A[6], k))
        e = hh * sum(c * v for c, v in zip(DP_E, k))
        err = (e.abs() / (tol + tol * torch.maximum(y0.abs(), xn.abs()))).amax(0)
        status[ids[~ok]] = 1
        worst = torch.zeros(G, dtype=torch.float64, device=x.device)
        worst.scatter_reduce_(0, gi[ok], err[ok], "amax")
        accept = worst <= 1.0
        take = ok & accept[gi]
        x[:, ids[take]] = xn[:, take]
        if left is not None:
            status[ids[take]] = torch.where(left(xn[:, take]), 1, 0).to(torch.uint8)
        any_ok = torch.zeros(G, dtype=torch.bool, device=x.device)
        any_ok[gi[ok]] = True
        f = torch.where(worst == 0, 5.0, (0.9 * worst.clamp(min=1e-300) ** -0.2).clamp(0.2, 5.0))
        t = torch.where(live_g & accept, torch.where(last, T, t + hs), t)
        h = torch.where(live_g & any_ok, hs * f, h)
    return x, status


def _gradient(case, x, status):
    """grad F [N][dim][dim] by lattice differences: central, else one-sided of second order, else NaN."""
    n, lo, hi, per = _lattice(case)
    dim = len(n)
    shape = tuple(n[::-1])
    ok = (status == 0).reshape(shape)
    G = torch.empty((x.shape[1], dim, dim), dtype=torch.float64, device=x.device)
    for b in range(dim):
        axis = dim - 1 - b
        h = (hi[b] - lo[b]) / (n[b] if per[b] else n[b] - 1)
        idx = torch.arange(n[b], device=x.device)

        def shifted(v, off, wrap):
            j = idx + off
            w = torch.div(j, n[b], rounding_mode="floor")
            r = v.index_select(axis, j % n[b])
            s = [1] * dim
            s[axis] = n[b]
            if not per[b]:
                return r, (w == 0).reshape(s)
            return (r + wrap * w.reshape(s), torch.ones(s, dtype=torch.bool, device=x.device))

        def good(off):
            o, inside = shifted(ok, off, 0) if not per[b] else (ok.index_select(axis, (idx + off) % n[b]), True)
            return o & inside

        p1, m1, p2, m2 = (good(o) for o in (1, -1, 2, -2))
        for a in range(dim):
            v = x[a].reshape(shape)
            wrap = (hi[b] - lo[b]) if a == b else 0.0
            vp1, vm1, vp2, vm2 = (shifted(v, o, wrap)[0] for o in (1, -1, 2, -2))
            d = torch.full(shape, float("nan"), dtype=torch.float64, device=x.device)
            d = torch.where(m1 & m2, (3.0 * v - 4.0 * vm1 + vm2) / (2 * h), d)
            d = torch.where(p1 & p2, (-3.0 * v + 4.0 * vp1 - vp2) / (2 * h), d)
            d = torch.where(p1 & m1, (vp1 - vm1) / (2 * h), d)
            G[:, a, b] = torch.where(ok, d, float("nan")).reshape(-1)
    return G


def _ftle(G, T):
    """(FTLE, C): the largest eigenvalue of C = G^T G in closed form (2D) or from its eigenvalues (3D)."""
    C = G.transpose(1, 2) @ G
    lam = torch.full((C.shape[0],), float("nan"), dtype=torch.float64, device=C.device)
    good = torch.isfinite(C).all(2).all(1)
    if C.shape[1] == 2:
        a, b, c = C[:, 0, 0], C[:, 0, 1], C[:, 1, 1]
        lam = 0.5 * (a + c) + torch.sqrt((0.5 * (a - c)) ** 2 + b * b)
    else:
        lam[good] = _eigh(C[good])[0][:, 2]
    return torch.log(lam) / (2.0 * abs(T)), C


def _eigh(C, sweeps=8):
    """Ascending eigenvalues [N][3] and eigenvectors [N][3 rows][3] of symmetric C by Jacobi rotations."""
    A = C.clone()
    V = torch.eye(3, dtype=torch.float64, device=C.device).expand_as(A).clone()
    for _ in range(sweeps):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            apq = A[:, p, q]
            tau = (A[:, q, q] - A[:, p, p]) / (2.0 * torch.where(apq == 0, 1.0, apq))
            t = torch.where(tau < 0, -1.0, 1.0) / (tau.abs() + torch.sqrt(1.0 + tau * tau))
            t = torch.where(apq == 0, 0.0, t)
            c = 1.0 / torch.sqrt(1.0 + t * t)
            s = (t * c)[:, None]
            c = c[:, None]
            for B in (A, V):
                bp, bq = B[:, :, p].clone(), B[:, :, q].clone()
                B[:, :, p], B[:, :, q] = c * bp - s * bq, s * bp + c * bq
            ap, aq = A[:, p].clone(), A[:, q].clone()
            A[:, p], A[:, q] = c * ap - s * aq, s * ap + c * aq
    ev, order = torch.diagonal(A, dim1=1, dim2=2).sort(dim=1)
    W = V.transpose(1, 2).gather(1, order[:, :, None].expand(-1, -1, 3))
    big = W.gather(2, W.abs().argmax(dim=2, keepdim=True))
    return ev, W * torch.where(big < 0, -1.0, 1.0)


def _packed(C):
    i, j = ((0, 0, 0, 1, 1, 2), (0, 1, 2, 1, 2, 2)) if C.shape[1] == 3 else ((0, 0, 1), (0, 1, 1))
    return C[:, i, j].contiguous()


def _network(P, xyt):
    """Pre-activations and outputs of the network in FP64 (parameters packed layer by layer)."""
    x, y, t = xyt.double()
    phi = torch.stack([x - MLP["center"][0], y - MLP["center"][1], torch.sin(MLP["omega"] * t),
                       torch.cos(MLP["omega"] * t), torch.sin(MLP["kx"] * x), torch.cos(MLP["kx"] * x),
                       torch.sin(MLP["ky"] * y)], 1)
    at, h = 0, phi
    for l, (o, i) in enumerate(((128, 7), (128, 128), (128, 128), (128, 128), (3, 128))):
        W, b = P[at:at + o * i].reshape(o, i), P[at + o * i:at + o * i + o]
        at += o * i + o
        z = h @ W.T + b
        h = z * torch.sigmoid(z) if l < 4 else z
    return h


def exact(case, seed):
    path = case["path"]
    if path == "network":
        P = torch.from_numpy(inputs.mlp_init(seed=seed)).to(DEV, torch.float64)
        pts = _points(case["n"], seed)
        return {"out": torch.cat([_network(P, c).T for c in pts.split(1 << 18, 1)], 1)}
    if path == "train":
        P = torch.from_numpy(inputs.mlp_init(seed=seed)).to(DEV, torch.float64).requires_grad_(True)
        xyt = _points(case["n"], seed)
        d, s, n = _displacements(xyt, seed).double(), MLP["out_scale"], case["n"]
        loss = 0.0
        for xc, dc in zip(xyt.split(1 << 15, 1), d.split(1 << 15, 1)):
            o = _network(P, xc)
            e = o[:, :2].T - dc / s
            miss = torch.log10(torch.linalg.vector_norm(s * o[:, :2].T - dc, dim=0) + 1e-7).detach()
            part = ((e * e).sum() + RHO_WEIGHT * ((o[:, 2] - miss) ** 2).sum()) / n
            part.backward()
            loss += float(part)
        g = P.grad
        return {"loss": loss, "grads": g, "params": P.detach() - LR * g / (g.abs() + 1e-8)}
    n = _lattice(case)[0]
    N, steps = math.prod(n), case.get("steps", 0)
    if path == "gyre":
        t0, Ts = _jobs(case)
        if N * sum(abs(T) / 0.05 for T in Ts) > EXACT_MOST_2D or sum(abs(T) / 0.05 for T in Ts) > 2000:
            return None
        frames, g = _gyre_field(case, seed)
        F, x0, out = _Rect(frames, g, case["storage"]), _lattice_points(case), []
        for t, T in zip(t0, Ts):
            x, st, _ = _rk4_rect(F, x0, t, T, 0.05)
            out.append(_ftle(_gradient(case, x, st), T)[0])
        return {"ftle": torch.stack(out)}
    if path.startswith("abc"):
        if N * steps * (3 if path == "abc_var" else 1) > EXACT_MOST_3D:
            return None
        frames, g = _abc_field(case, seed)
        F, x0, T = _Rect(frames, g, case["storage"]), _lattice_points(case), 0.02 * case["steps"]
        M = torch.eye(3, dtype=torch.float64, device=DEV).expand(N, 3, 3) if path == "abc_var" else None
        x, st, M = _rk4_rect(F, x0, 0.0, T, 0.02, M)
        if path == "abc_var":
            return {"ftle": _ftle(M, T)[0][None], "grad": M}
        G = _gradient(case, x, st)
        if path == "abc_eigen":
            ev, W = _eigh(G.transpose(1, 2) @ G)
            return {"eigval": ev, "eigvec": W}
        s, C = _ftle(G, T)
        return {"ftle": s[None], "C": _packed(C)}
    x0 = _lattice_points(case)
    status = torch.zeros(N, dtype=torch.uint8, device=DEV)
    if path == "gyre_rk45":
        if N > 4000000:
            return None
        frames, g = _gyre_field(case, seed)
        F, times = _Rect(frames, g, case["storage"]), torch.from_numpy(g["times"]).to(DEV)

        def evaluate(y, ids, t):
            t = t - 10.0 * torch.floor(t / 10.0)
            k = (torch.searchsorted(times, t, right=True) - 1).clamp(0, 99)
            return F.at(y, k, (t - times[k]) / (times[k + 1] - times[k]))

        T = case["t_long"]
        x, status = _rk45(evaluate, F.left, x0, status, T, 0.05)
        return {"ftle": _ftle(_gradient(case, x, status), T)[0][None], "xyz": x}
    if N * (steps or 80) > EXACT_MOST_MESH:
        return None
    frames, g = FIELDS[path](case, seed)
    F = _Mesh(frames, g, case["storage"])
    if path == "stenosis":
        start = (x0[1].abs() <= _halfwidth(x0[0], g["extra"])[0]).logical_not()   # beside the constriction
        i = (x0[0] / case["h"]).long().clamp(0, int(round(10 / case["h"])) - 1)
        s = x0[1] / _halfwidth(x0[0], g["extra"])[0]
        j = ((s.clamp(-1, 1) + 1.0) / case["h"]).long().clamp(0, 2 * int(round(1 / case["h"])) - 1)
        cell = 2 * (i + int(round(10 / case["h"])) * j)
        cell, inside = F.locate(torch.where(start, torch.zeros_like(x0) + 5.0 * torch.tensor([[1.0], [0.0]], device=DEV),
                                            x0), cell)
        status[start | ~inside] = 2
        T, dt = 0.002 * steps, 0.002
    else:
        m = case["m"]
        i, j = (((x0[d] + 1.0) * m).long().clamp(0, 2 * m - 1) for d in (0, 1))
        k = (x0[2] * m).long().clamp(0, 10 * m - 1)
        cell, inside = F.locate(x0, 6 * (i + 2 * m * (j + 2 * m * k)))
        status[~inside] = 2
        T, dt = (1.0, None) if path == "duct_rk45" else (0.01 * steps, 0.01)
    if dt is None:
        nodes, flat = F.F.shape[1], F.F.reshape(-1, 3)

        def evaluate(y, ids, t):
            cl, inside = F.locate(y, cell[ids])
            cell[ids] = cl
            t = t - torch.floor(t)
            k = (t * 50.0).long().clamp(0, 49)
            a = (t * 50.0 - k)[:, None, None]
            v = F.cells[cl] + (k * nodes)[:, None]
            u = (1.0 - a) * flat[v].double() + a * flat[v + nodes].double()
            return torch.einsum("ni,nid->dn", F.bary(cl, y), u), inside

        x, status = _rk45(evaluate, None, x0, status, T, 0.02)
    else:
        x, status = _rk4_mesh(F, x0, cell, status, T, dt)
    return {"ftle": _ftle(_gradient(case, x, status), T)[0][None], "xyz": x}
