"""Both layouts of the 3D time slices (quads on dense lattices, plain nodes on sparse ones) against the one-pass
kernels, bit for bit: tracer densities on both sides of the rule, odd node counts, mixed periodicity, storage
types, snapshots, and the variational equations on a lattice dense enough for quads otherwise."""
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


def flow_map(ctx, field, seeds, N, variant, variational):
    nslot = 1 if variational else 3
    fm = lcs.lcs_flowmap_create(ctx, seeds, nslot)
    o = lcs.advect_opts(lcs.RK4, t0=0.05, T=0.5, dt=0.02, variant=variant, episode_steps=6,
                        snap_T=None if variational else [0.1, 0.26], variational=variational)
    lcs.lcs_advect(ctx, field, seeds, o, fm)
    out = []
    for j in range(nslot):
        x, s, t = np.empty((3, N), np.float32), np.empty(N, np.uint8), np.empty(N, np.float32)
        lcs.lcs_flowmap_get(ctx, fm, j, x, s, t)
        out += [x, s, t]
    if variational:
        M = np.empty((N, 3, 3), np.float32)
        lcs.lcs_flowmap_grad(ctx, fm, 0, M)
        out.append(M)
    lcs.lcs_free_flowmap(fm)
    return out


@pytest.mark.parametrize("variational", [False, True])
@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 0, 0), (0, 1, 0)])
@pytest.mark.parametrize("grid,n,storage", [(5, (9, 8, 7), lcs.F32), (5, (10, 10, 9), lcs.BF16), (9, (11, 3, 5), lcs.F32),
                                            (16, (29, 29, 29), lcs.F16), (16, (30, 29, 29), lcs.F32)])
def test_layouts_equal_one_pass(ctx, grid, n, storage, periodic, variational):
    from dataclasses import replace
    g = replace(inputs.abc(n=grid, nframes=4, t_end=1.0), periodic=periodic)
    field = lcs.lcs_load_field(ctx, rect_desc(g, storage), g.frames)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(3, n, (0.1, 0.2, 0.3), (5.9, 5.5, 5.8)))
    N = lcs.lcs_seeds_count(seeds)
    try:
        for a, b in zip(flow_map(ctx, field, seeds, N, 1, variational), flow_map(ctx, field, seeds, N, 3, variational)):
            np.testing.assert_array_equal(a, b)
    finally:
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_field(field)
