"""RK4 on triangles by both forms of its kernel: lattices on either side of the dispatch's tracer count whose first rows
hold the same seeds, every storage type, one job and a job count that crosses the line, bit for bit."""
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
def channel():
    mesh = inputs.stenosis_mesh(h=0.04)
    return inputs.stenosis_frames(mesh, nframes=10, period=1.0)


def flow_map(ctx, field, rows, njobs):
    # positions exact in FP32: steps of 1/32 along x and 1/1024 along y
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(2, (256, rows), (0.5, -0.25), (0.5 + 255 / 32, -0.25 + (rows - 1) / 1024)),
                              field)
    N = lcs.lcs_seeds_count(seeds)
    fm = lcs.lcs_flowmap_create(ctx, seeds, njobs)
    lcs.lcs_advect(ctx, field, seeds, lcs.advect_opts(lcs.RK4, dt=0.01, job_t0=[0.1] * njobs, job_T=[0.6] * njobs), fm)
    x, s, t = np.empty((2, N), np.float32), np.empty(N, np.uint8), np.empty(N, np.float32)
    lcs.lcs_flowmap_get(ctx, fm, njobs - 1, x, s, t)
    lcs.lcs_free_flowmap(fm)
    lcs.lcs_free_seeds(seeds)
    return x, s, t


@pytest.mark.parametrize("storage", [lcs.F32, lcs.F16, lcs.BF16])
def test_both_forms(ctx, channel, storage):
    g = channel
    field = lcs.lcs_load_field(ctx, lcs.field_desc(2, times=g.times, time_periodic=True, period=g.period, storage=storage,
                                                   kind=lcs.TRI, mesh=(g.xyz, g.tets, g.nbrs)), g.frames)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    try:
        x, s, t = flow_map(ctx, field, 37, 1)
        n = s.size
        for rows, njobs in ((2 * sms, 1), (2 * sms + 1, 1), (37, 9)):
            xb, sb, tb = flow_map(ctx, field, rows, njobs)
            np.testing.assert_array_equal(xb[:, :n], x)
            np.testing.assert_array_equal(sb[:n], s)
            np.testing.assert_array_equal(tb[:n], t)
    finally:
        lcs.lcs_free_field(field)
