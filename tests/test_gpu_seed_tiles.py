"""Warps that take blocks of the seed lattice give what warps that take consecutive seeds give, bit for bit:
every one-thread-per-tracer kernel, lattices with ragged edges, snapshots, tracers that leave.  A block size
that is no multiple of 32 keeps the consecutive order, so it serves as the other side."""
import numpy as np
import pytest
import torch

from gpu_util import rect_desc
from meshes import kuhn_mesh
from paper_2209_13775_gb300 import inputs, lcs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


def field_of(ctx, kind):
    if kind == "gyre":
        g = inputs.double_gyre(nx=33, ny=17, nframes=11, t_end=1.0)
        return lcs.lcs_load_field(ctx, rect_desc(g), g.frames), (-0.3, 0.0), (1.6, 1.2)
    if kind == "abc":
        g = inputs.abc(n=16, nframes=5, t_end=1.0)
        return lcs.lcs_load_field(ctx, rect_desc(g, lcs.BF16), g.frames), (0.0, 0.5, 0.2), (5.0, 6.0, 4.0)
    if kind == "tri":
        m = inputs.stenosis_frames(inputs.stenosis_mesh(h=0.2), nframes=5)
        lo, hi = (0.1, -0.9), (9.9, 0.9)
    else:
        xyz, tets, nbrs = kuhn_mesh(4)
        m = inputs.TetInput(xyz, tets, nbrs)
        m.times, m.period = np.array([0.0, 0.5, 1.0]), 1.0
        rng = np.random.default_rng(1)
        m.frames = rng.uniform(-3, 3, (3, xyz.shape[0], 3)).astype(np.float32)
        lo, hi = (0.1, 0.2, 0.0), (3.9, 4.0, 3.7)
    d = lcs.field_desc(len(lo), times=m.times, time_periodic=True, period=m.period,
                       kind=lcs.TRI if kind == "tri" else lcs.TET, mesh=(m.xyz, m.tets, m.nbrs))
    return lcs.lcs_load_field(ctx, d, m.frames), lo, hi


def outputs(ctx, field, seeds, N, dim, bt, variant, variational):
    njobs = 1 if variational else 2
    snaps = None if variational else [0.1, 0.4]
    fm = lcs.lcs_flowmap_create(ctx, seeds, njobs * (1 if variational else 3))
    o = lcs.advect_opts(lcs.RK4, dt=0.05, job_t0=[0.1, 0.3][:njobs], job_T=[0.6, -0.4][:njobs], variant=variant,
                        block_threads=bt, snap_T=snaps, variational=variational)
    lcs.lcs_advect(ctx, field, seeds, o, fm)
    out = []
    for j in range(njobs * (1 if variational else 3)):
        x, s, t = np.empty((dim, N), np.float32), np.empty(N, np.uint8), np.empty(N, np.float32)
        lcs.lcs_flowmap_get(ctx, fm, j, x, s, t)
        out += [x, s, t]
    if variational:
        M = np.empty((N, dim, dim), np.float32)
        lcs.lcs_flowmap_grad(ctx, fm, 0, M)
        out.append(M)
    lcs.lcs_free_flowmap(fm)
    return out


@pytest.mark.parametrize("variational", [False, True])
@pytest.mark.parametrize("kind,n", [("gyre", (16, 16)), ("gyre", (33, 31)), ("gyre", (170, 14)), ("gyre", (300, 3)),
                                    ("tri", (45, 16)), ("tri", (129, 31)), ("abc", (8, 8, 4)), ("abc", (23, 15, 11)),
                                    ("tet", (16, 7, 12)), ("tet", (39, 23, 3))])
def test_tiled_equals_linear(ctx, kind, n, variational):
    field, lo, hi = field_of(ctx, kind)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(len(n), n, lo, hi), field)
    N = lcs.lcs_seeds_count(seeds)
    try:
        for variant in ((1, 5) if kind == "gyre" and not variational else (1,)):
            a = outputs(ctx, field, seeds, N, len(n), 100, variant, variational)
            for bt in (0, 32, 96):
                b = outputs(ctx, field, seeds, N, len(n), bt, variant, variational)
                for u, v in zip(a, b):
                    np.testing.assert_array_equal(u, v)
    finally:
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_field(field)
