"""The phases that lcs_timing_read reports for the 2D time slices: the fill and the advection, one launch each, asked
for (variant 5) and by default, and a second read that finds nothing new."""
import pytest
import torch

from gpu_util import rect_desc
from paper_2209_13775_gb300 import inputs, lcs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 5])
def test_slice_phases(variant):
    torch.cuda.set_device(0)
    ctx = lcs.lcs_create(0, torch.cuda.current_stream())
    g = inputs.double_gyre(nx=33, ny=17, nframes=11, t_end=1.0)
    field = lcs.lcs_load_field(ctx, rect_desc(g), g.frames)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(2, (64, 32), (0.0, 0.0), (2.0, 1.0)))
    fm = lcs.lcs_flowmap_create(ctx, seeds, 2)
    try:
        lcs.lcs_timing_enable(ctx, True)
        lcs.lcs_advect(ctx, field, seeds, lcs.advect_opts(lcs.RK4, dt=0.05, job_t0=[0.0, 0.1], job_T=[0.5, 0.8],
                                                          variant=variant), fm)
        for phase in (lcs.PHASE_ADVECT, lcs.PHASE_SLICES):
            ms, launches = lcs.lcs_timing_read(ctx, phase)
            assert launches == 1 and 0.0 < ms < 1000.0, (phase, ms, launches)
            assert lcs.lcs_timing_read(ctx, phase) == (0.0, 0)
        assert lcs.lcs_timing_read(ctx, lcs.PHASE_REBUNDLE) == (0.0, 0)
        lcs.lcs_timing_enable(ctx, False)
    finally:
        lcs.lcs_free_flowmap(fm)
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_field(field)
        lcs.lcs_destroy(ctx)
