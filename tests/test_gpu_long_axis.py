"""All-periodic 3D boxes with an axis of 2^21 to 2^22 nodes, where an FP32 coordinate in cells reaches 2^22 and more
within a period of the box: one RK4 step whose stages pass the end of that axis by one to a thousand cells, one-pass
and re-bundled, against the FP64 oracle.

u_x = 2, and u_y rises by 2^-12 from node to node over runs of 1024 nodes, constant along y and z; seeds and stage
points lie on nodes of the long axis, so a stage that reads the next cell is off by 2^-12 in u_y, by dt 2^-12 / 6
in y at the least.  Rounding: y and the sum of eight weighted slopes, 16 ulps of (3 + dt) at the most; x is exact to
the spacing of FP32 there, 0.5."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import oracle_field, rect_desc
from paper_2209_13775_gb300 import inputs, lcs

pytestmark = pytest.mark.gpu
SLOPE = 2.0 ** -12


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


@pytest.mark.parametrize("n0", [2 ** 21, 2 ** 21 + 4, 2 ** 22 - 4, 2 ** 22])
def test_stages_past_the_end(ctx, n0):
    frames = np.zeros((1, 3, 3, n0, 3), np.float32)
    frames[..., 0] = 2.0
    frames[..., 1] = (SLOPE * (np.arange(n0) % 1024)).astype(np.float32)
    g = inputs.RectInput(frames, np.zeros(1), (0.0,) * 3, (1.0,) * 3, (1, 1, 1))
    n, lo, hi = (128, 2, 2), (n0 - 128.0, 0.0, 0.25), (n0 - 1.0, 1.25, 2.0)
    x0 = oracle.seed_grid(3, n, lo, hi, [1, 1, 1]).astype(np.float64)
    F = oracle_field(g)
    field = lcs.lcs_load_field(ctx, rect_desc(g), frames)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(3, n, lo, hi))
    fm = lcs.lcs_flowmap_create(ctx, seeds, 1)
    try:
        for dt in (1.0, 2.0, 3.0, 8.0, 50.0, 500.0):
            xo, so, _ = oracle.rk4(F, x0, 0.0, dt, dt)
            got = []
            for variant, var in ((1, False), (1, True), (3, False), (3, True)):
                x, s = np.empty(x0.shape, np.float32), np.empty(x0.shape[1], np.uint8)
                lcs.lcs_advect(ctx, field, seeds, lcs.advect_opts(lcs.RK4, T=dt, dt=dt, variant=variant, variational=var,
                                                                  episode_steps=1), fm)
                lcs.lcs_flowmap_get(ctx, fm, 0, x, s)
                np.testing.assert_array_equal(s, so)
                got.append(x)
            for x in got:
                assert np.abs(x[0] - xo[0]).max() <= 0.5
                assert np.abs(x[1] - xo[1]).max() <= 16 * 2.0 ** -24 * (3 + dt), (dt, np.abs(x[1] - xo[1]).max())
                np.testing.assert_array_equal(x, got[0])
    finally:
        lcs.lcs_free_flowmap(fm)
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_field(field)
