"""Where the default of 3D boxes goes over to re-bundled episodes: boxes periodic along some axes only do at half the
tracers that all-periodic and closed ones take (rk4_rebundle_seeds; 125 nodes, 17 steps), and both sides of the line
give the positions of either variant bit for bit."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from gpu_util import rect_desc
from paper_2209_13775_gb300 import inputs, lcs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("periodic,n,rebundled", [
    ((1, 0, 1), (64, 64, 64), False), ((1, 0, 1), (65, 65, 64), True), ((0, 1, 0), (65, 65, 64), True),
    ((1, 1, 1), (65, 65, 64), False), ((0, 0, 0), (65, 65, 64), False), ((1, 1, 1), (81, 81, 80), True)])
def test_default_choice(periodic, n, rebundled):
    torch.cuda.set_device(0)
    ctx = lcs.lcs_create(0, torch.cuda.current_stream())
    g = replace(inputs.abc(n=5, nframes=3, t_end=1.0), periodic=periodic)
    field = lcs.lcs_load_field(ctx, rect_desc(g), g.frames)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(3, n, (0.1, 0.1, 0.1), (4.8, 4.8, 4.8)))
    N = lcs.lcs_seeds_count(seeds)
    fm = lcs.lcs_flowmap_create(ctx, seeds, 1)
    out = []
    try:
        lcs.lcs_timing_enable(ctx, True)
        for variant in (0, 1, 3):
            lcs.lcs_advect(ctx, field, seeds, lcs.advect_opts(lcs.RK4, T=0.34, dt=0.02, variant=variant), fm)
            assert (lcs.lcs_timing_read(ctx, lcs.PHASE_REBUNDLE)[1] > 0) == (rebundled if variant == 0 else variant == 3)
            x, s = np.empty((3, N), np.float32), np.empty(N, np.uint8)
            lcs.lcs_flowmap_get(ctx, fm, 0, x, s)
            out.append((x, s))
        for x, s in out[1:]:
            np.testing.assert_array_equal(x, out[0][0])
            np.testing.assert_array_equal(s, out[0][1])
        lcs.lcs_timing_enable(ctx, False)
    finally:
        lcs.lcs_free_flowmap(fm)
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_field(field)
        lcs.lcs_destroy(ctx)
