"""The 2D time-slice kernel of closed boxes against the cached-gather kernel, bit for bit: boxes whose last
fraction is and is not exactly 1, origins off zero, one and many frames, start times off and on the frames
(first slices shared with the step before, or not), backward jobs, tracers that leave, snapshots."""
import numpy as np
import pytest
import torch

from paper_2209_13775_gb300 import lcs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


@pytest.mark.parametrize("lattice", [(61, 37), (331, 151)])   # records copied ahead (few tracers), and not
@pytest.mark.parametrize("storage", [lcs.F32, lcs.BF16])
@pytest.mark.parametrize("nf,time_periodic", [(1, False), (2, False), (9, True)])
@pytest.mark.parametrize("n,origin,spacing", [((2, 2), (0.0, 0.0), (1.0, 0.5)), ((17, 9), (-0.3, 1.7), (0.1, 0.07)),
                                              ((129, 65), (0.0, 0.0), (2 / 128, 1 / 64)),
                                              ((40, 31), (1e3, -7.0), (0.3, 1 / 3))])
def test_slices_equal_gather(ctx, n, origin, spacing, nf, time_periodic, storage, lattice):
    rng = np.random.default_rng(n[0] + nf)
    frames = (rng.standard_normal((nf, n[1], n[0], 2)) * np.array(spacing) * 4).astype(np.float32)
    d = lcs.field_desc(2, n=n, origin=origin, spacing=spacing, times=np.arange(nf) * 0.25,
                       time_periodic=time_periodic, period=nf * 0.25, storage=storage)
    field = lcs.lcs_load_field(ctx, d, frames)
    hi = [origin[a] + (n[a] - 1) * spacing[a] for a in range(2)]
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(2, lattice, [o - 0.4 * s for o, s in zip(origin, spacing)],
                                                 [h + 0.4 * s for h, s in zip(hi, spacing)]))
    N, got = lcs.lcs_seeds_count(seeds), []
    try:
        for variant in (1, 5):
            fm = lcs.lcs_flowmap_create(ctx, seeds, 9)
            o = lcs.advect_opts(lcs.RK4, dt=0.05, job_t0=[0.0, 0.13, 1.0], job_T=[1.0, 0.35, -0.8],
                                snap_T=[0.05, 0.35], variant=variant)
            lcs.lcs_advect(ctx, field, seeds, o, fm)
            out = []
            for j in range(9):
                x, s, t = np.empty((2, N), np.float32), np.empty(N, np.uint8), np.empty(N, np.float32)
                lcs.lcs_flowmap_get(ctx, fm, j, x, s, t)
                out += [x, s, t]
            lcs.lcs_free_flowmap(fm)
            got.append(out)
    finally:
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_field(field)
    assert any((s != 0).any() for s in got[0][1::3])   # some tracers leave
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


def test_more_runs_than_grid_rows(ctx):
    # 300,000 steps on a 2 x 2 grid: the fill's runs of slices exceed a grid's 65,535 rows
    frames = np.array([[[[0.1, -0.2], [0.05, 0.1]], [[-0.1, 0.2], [0.15, -0.1]]]], dtype=np.float32)
    d = lcs.field_desc(2, n=(2, 2), origin=(0, 0), spacing=(1, 1), times=[0.0])
    field = lcs.lcs_load_field(ctx, d, frames)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(2, (3, 3), (0.2, 0.2), (0.8, 0.8)))
    got = []
    for variant in (1, 5):
        fm = lcs.lcs_flowmap_create(ctx, seeds, 1)
        lcs.lcs_advect(ctx, field, seeds, lcs.advect_opts(lcs.RK4, T=3.0, dt=1e-5, variant=variant), fm)
        x = np.empty((2, 9), np.float32)
        lcs.lcs_flowmap_get(ctx, fm, 0, x)
        lcs.lcs_free_flowmap(fm)
        got.append(x)
    lcs.lcs_free_seeds(seeds)
    lcs.lcs_free_field(field)
    np.testing.assert_array_equal(*got)
