"""The 3D one-pass kernels against the re-bundled episodes, bit for bit: every box kind of the cell search (all axes
periodic, all closed, mixed), axes of three nodes and more, seeds many periods away from the box, steps across several
periods, coarse frames (many stages per cell) and frames finer than a step, several jobs, plain positions and
variational gradients, and the default choice on both sides of its rule."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from gpu_util import rect_desc
from paper_2209_13775_gb300 import inputs, lcs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


def flow_maps(ctx, field, seeds, variant, block=0, variational=False, dt=0.02, njobs=2):
    N = lcs.lcs_seeds_count(seeds)
    fm = lcs.lcs_flowmap_create(ctx, seeds, njobs)
    o = lcs.advect_opts(lcs.RK4, dt=dt, job_t0=[0.05, 0.3][:njobs], job_T=[0.5, 0.34][:njobs], variant=variant,
                        block_threads=block, variational=variational)
    lcs.lcs_advect(ctx, field, seeds, o, fm)
    out = []
    for j in range(njobs):
        x, s, t = np.empty((3, N), np.float32), np.empty(N, np.uint8), np.empty(N, np.float32)
        lcs.lcs_flowmap_get(ctx, fm, j, x, s, t)
        out += [x, s, t]
        if variational:
            out.append(np.empty((N, 3, 3), np.float32))
            lcs.lcs_flowmap_grad(ctx, fm, j, out[-1])
    lcs.lcs_free_flowmap(fm)
    return out


@pytest.mark.parametrize("variational", [False, True])
@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 0, 0), (1, 0, 1)])
@pytest.mark.parametrize("grid,nframes,storage,block,speed", [
    (3, 2, lcs.F32, 64, 1.0), (4, 40, lcs.F16, 0, 1.0), (11, 5, lcs.BF16, 32, 300.0), (17, 90, lcs.F32, 256, 1.0)])
def test_equals_episodes(ctx, grid, nframes, storage, block, speed, periodic, variational):
    g = inputs.abc(n=grid, nframes=nframes, t_end=1.0)
    g = replace(g, periodic=periodic, frames=np.float32(speed) * g.frames)
    field = lcs.lcs_load_field(ctx, rect_desc(g, storage), g.frames)
    h = [float(v) for v in g.spacing]
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(3, (13, 7, 9), (-20.0, 0.1, -40.0), (26.0, 2e4, 45.0)))
    seeds2 = lcs.lcs_seed_grid(ctx, lcs.seed_desc(3, (10, 11, 9), (0.02, 0.05, 0.1), tuple(h[d] * grid * 0.99 for d in range(3))))
    try:
        for sd in (seeds, seeds2):
            a = flow_maps(ctx, field, sd, 1, block, variational)
            b = flow_maps(ctx, field, sd, 3, 0, variational)
            for u, v in zip(a, b):
                np.testing.assert_array_equal(u, v)
    finally:
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_seeds(seeds2)
        lcs.lcs_free_field(field)


@pytest.mark.parametrize("variational", [False, True])
@pytest.mark.parametrize("n", [(80, 81, 80), (81, 81, 80)])
def test_default_rule(ctx, n, variational):
    g = inputs.abc(n=5, nframes=3, t_end=1.0)
    field = lcs.lcs_load_field(ctx, rect_desc(g, lcs.F32), g.frames)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(3, n, (0.0, 0.0, 0.0), (6.0, 6.0, 6.0)))
    try:
        a = flow_maps(ctx, field, seeds, 0, 0, variational, njobs=1)
        for variant in (1, 3):
            for u, v in zip(a, flow_maps(ctx, field, seeds, variant, 0, variational, njobs=1)):
                np.testing.assert_array_equal(u, v)
    finally:
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_field(field)
