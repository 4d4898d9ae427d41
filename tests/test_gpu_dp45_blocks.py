"""DP5(4) on tets by both register splits of its kernel: lattices on either side of the dispatch's tracer count whose
first layers hold the same seeds (so the same warps), every storage type, one job and a job count that crosses the line,
bit for bit."""
import numpy as np
import pytest
import torch

from paper_2209_13775_gb300 import inputs, lcs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


@pytest.fixture(scope="module")
def pipe():
    return inputs.pipe_frames(inputs.pipe_mesh(h=0.15, R=1.0, L=2.0), nframes=20, period=1.0, L=2.0)


def flow_map(ctx, field, layers, njobs):
    # positions exact in FP32: 32 x 32 seeds at steps of 1/32, layers at steps of 1/256
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(3, (32, 32, layers), (-0.5, -0.5, 0.25),
                                                 (15 / 32, 15 / 32, 0.25 + (layers - 1) / 256)), field)
    N = lcs.lcs_seeds_count(seeds)
    fm = lcs.lcs_flowmap_create(ctx, seeds, njobs)
    o = lcs.advect_opts(lcs.RK45, job_t0=[0.1] * njobs, job_T=[0.7] * njobs, rtol=1e-5, atol=1e-5)
    lcs.lcs_advect(ctx, field, seeds, o, fm)
    x, s, t = np.empty((3, N), np.float32), np.empty(N, np.uint8), np.empty(N, np.float32)
    lcs.lcs_flowmap_get(ctx, fm, njobs - 1, x, s, t)
    lcs.lcs_free_flowmap(fm)
    lcs.lcs_free_seeds(seeds)
    return x, s, t


@pytest.mark.parametrize("storage", [lcs.F32, lcs.F16, lcs.BF16])
def test_both_splits(ctx, pipe, storage):
    field = lcs.lcs_load_field(ctx, lcs.field_desc(3, times=pipe.times, time_periodic=True, period=pipe.period,
                                                   storage=storage, kind=lcs.TET,
                                                   mesh=(pipe.xyz, pipe.tets, pipe.nbrs)), pipe.frames)
    try:
        x, s, t = flow_map(ctx, field, 64, 1)          # 65,536 tracers: three blocks
        n = s.size
        for layers, njobs in ((255, 1), (256, 1), (64, 4)):   # 261,120; 262,144 twice: four in 16 bits
            xb, sb, tb = flow_map(ctx, field, layers, njobs)
            np.testing.assert_array_equal(xb[:, :n], x)
            np.testing.assert_array_equal(sb[:n], s)
            np.testing.assert_array_equal(tb[:n], t)
    finally:
        lcs.lcs_free_field(field)
