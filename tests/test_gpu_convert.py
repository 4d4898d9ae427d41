"""Frames into storage: frame counts around the run of slabs one thread stores, single frames, odd node counts, each
layout (2D, 3D interval pairs, triangle pairs) and type; the stored values read back through one
step of a velocity constant in space, and a non-finite value in any frame refused."""
import numpy as np
import pytest
import torch

from paper_2209_13775_gb300 import lcs

pytestmark = pytest.mark.gpu
ROUND = {lcs.F32: lambda v: v, lcs.F16: lambda v: v.astype(np.float16).astype(np.float32),
         lcs.BF16: lambda v: torch.from_numpy(v).bfloat16().float().numpy()}


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


@pytest.mark.parametrize("storage", [lcs.F32, lcs.F16, lcs.BF16])
@pytest.mark.parametrize("nframes", [1, 2, 3, 4, 5, 6, 8, 9, 10, 17])
@pytest.mark.parametrize("n", [(17, 19), (7, 6, 9)])
def test_rect_frames(ctx, n, nframes, storage):
    """Seeds on the nodes, one Euler-sized step at every frame time: x(h) - x = h u(node) for a field that is constant
    in space, so the displacement is the stored frame value (weights sum to 1 in FP32 within 2^-22)."""
    dim = len(n)
    rng = np.random.default_rng(nframes)
    vals = rng.uniform(0.5, 1.5, size=(nframes, dim)).astype(np.float32)
    frames = np.ascontiguousarray(np.broadcast_to(vals.reshape((nframes,) + (1,) * dim + (dim,)),
                                                  (nframes,) + n[::-1] + (dim,)))
    times = np.arange(nframes, dtype=np.float64)
    desc = lcs.field_desc(dim, n, (0.0,) * dim, (1.0,) * dim, (1,) * dim, times, False, 0.0, storage=storage)
    field = lcs.lcs_load_field(ctx, desc, frames)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(dim, (3,) * dim, (1.0,) * dim, (2.0,) * dim))
    N = lcs.lcs_seeds_count(seeds)
    want = ROUND[storage](vals)
    try:
        for k in range(nframes - 1):
            fm = lcs.lcs_flowmap_create(ctx, seeds, 1)
            lcs.lcs_advect(ctx, field, seeds, lcs.advect_opts(lcs.RK4, t0=float(k), T=1.0, dt=1.0, variant=1), fm)
            x, s, t = np.empty((dim, N), np.float32), np.empty(N, np.uint8), np.empty(N, np.float32)
            lcs.lcs_flowmap_get(ctx, fm, 0, x, s, t)
            lcs.lcs_free_flowmap(fm)
            mean = 0.5 * (want[k].astype(np.float64) + want[k + 1])   # RK4 of a velocity linear in time
            # x < 4: positions to 2^-22, stage velocities to 2^-22 of 1.5
            np.testing.assert_allclose(x[:, 0], 1.0 + mean, rtol=0, atol=4 * 2.0 ** -22)
    finally:
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_free_field(field)


@pytest.mark.parametrize("n", [(17, 19), (7, 6, 9)])
def test_nonfinite_any_frame(ctx, n):
    dim = len(n)
    for nframes in (1, 4, 5, 9):
        for k in range(nframes):
            frames = np.zeros((nframes,) + n[::-1] + (dim,), np.float32)
            frames[k].reshape(-1)[-1 - k] = np.inf if k % 2 else np.nan
            desc = lcs.field_desc(dim, n, (0.0,) * dim, (1.0,) * dim, (1,) * dim, np.arange(nframes, dtype=np.float64),
                                  False, 0.0, storage=lcs.F32)
            with pytest.raises(lcs.LcsError):
                lcs.lcs_load_field(ctx, desc, frames)
