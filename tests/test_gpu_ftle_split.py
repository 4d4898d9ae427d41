"""The FTLE in double-FP32 and the two-operation division by 2h, against the FP64 oracle on the same
positions: every difference rule, periodic and bounded lattices, spacings and magnitudes on both sides of
the range the split arithmetic takes, equal eigenvalues, infinite and NaN positions.

C is bit-identical to the oracle's.  sigma = ln(lambda) / (2 |T|) is rounded to FP32 by a logarithm (2 ulps),
the factor 1 / (2 |T|) and their product (half an ulp each): 3 ulps of 2^-23 relative, plus the eigenvalue's
own error, 2^-40 relative (1e-9 where the two largest coincide), over 2 |T|.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2209_13775_gb300 import lcs

pytestmark = pytest.mark.gpu
T = 1.75
RTOL = 3 * 2.0 ** -23


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


def both(ctx, n, lo, hi, periodic, x, st):
    """(FTLE alone, FTLE with lambda and C, C) of the library and (C, sigma) of the oracle."""
    dim = len(n)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(dim, n, lo, hi, periodic))
    fm = lcs.lcs_flowmap_create(ctx, seeds, 1)
    N = int(np.prod(n))
    f, g, lam, C = (np.empty(N, np.float32), np.empty(N, np.float32), np.empty(N),
                    np.empty((N, 3 if dim == 2 else 6)))
    try:
        lcs.lcs_flowmap_set(ctx, fm, 0, x, st, T)
        lcs.lcs_ftle(ctx, fm, 0, f)
        lcs.lcs_ftle(ctx, fm, 0, g, lam, C)
    finally:
        lcs.lcs_free_flowmap(fm)
        lcs.lcs_free_seeds(seeds)
    h = oracle.lattice_spacing(dim, n, lo, hi, [0 if p else 1 for p in periodic])
    period = [hi[a] - lo[a] if periodic[a] else 0.0 for a in range(dim)]
    with np.errstate(all="ignore"):
        Co = oracle.cauchy_green(oracle.flowmap_gradient(dim, n, h, periodic, period, x.astype(np.float64), st))
        sig = oracle.ftle(Co, dim, T)[1]
    np.testing.assert_array_equal(f, g)   # the FTLE does not depend on the other outputs
    return f, C, Co, sig


@pytest.mark.parametrize("scale", [1e-16, 1e-12, 1e-3, 1.0, 1e4, 1e15])
@pytest.mark.parametrize("n", [(3, 3), (33, 17), (257, 4), (3, 3, 3), (33, 5, 4), (64, 9, 3)])
@pytest.mark.parametrize("per", [0, 1])
def test_random_positions(ctx, n, per, scale):
    rng = np.random.default_rng(len(n) * 1000 + n[0] + per)
    dim, N = len(n), int(np.prod(n))
    lo, hi = tuple(0.1 * scale for _ in n), tuple(scale * (0.1 + 0.7 * (a + 1)) for a in range(dim))
    x = (rng.standard_normal((dim, N)) * 0.5).astype(np.float32)
    st = np.where(rng.random(N) < 0.15, oracle.LEFT, 0).astype(np.uint8)
    f, C, Co, sig = both(ctx, n, lo, hi, (per,) * dim, x, st)
    np.testing.assert_array_equal(C, Co)
    ok = np.isfinite(sig)
    np.testing.assert_array_equal(np.isfinite(f), ok)
    np.testing.assert_allclose(f[ok], sig[ok], rtol=RTOL, atol=2.0 ** -40 / T)


@pytest.mark.parametrize("dim", [2, 3])
def test_equal_and_nearly_equal_eigenvalues(ctx, dim):
    # x = k times the lattice positions: C = k^2 I; a shear of the last axis then splits the eigenvalues
    n = (12, 11, 10)[:dim]
    lo, hi = (0.0,) * dim, (1.1,) * dim
    grid = np.stack([a.ravel() for a in np.meshgrid(*[np.linspace(0, 1.1, m) for m in n[::-1]],
                                                    indexing="ij")[::-1]])
    for k in (1.0, 0.37, 21.0):
        for shear in (0.0, 1e-7, 1e-5, 1e-3, 0.1):
            x = k * grid
            x[0] = x[0] + shear * grid[dim - 1]
            if dim == 3:
                x[2] *= 0.5   # the two largest (nearly) equal, the smallest apart
            x = x.astype(np.float32)
            f, C, Co, sig = both(ctx, n, lo, hi, (0,) * dim, x, np.zeros(x.shape[1], np.uint8))
            np.testing.assert_array_equal(C, Co)
            np.testing.assert_allclose(f, sig, rtol=RTOL, atol=1e-9)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_positions(ctx, bad):
    n = (9, 8, 7)
    rng = np.random.default_rng(3)
    x = rng.standard_normal((3, 9 * 8 * 7)).astype(np.float32)
    x[1, 200] = bad
    f, C, Co, sig = both(ctx, n, (0.0,) * 3, (1.0, 2.0, 3.0), (0, 0, 0), x, np.zeros(x.shape[1], np.uint8))
    touched = ~np.isfinite(sig)
    assert 6 <= touched.sum() <= 8 and not np.isfinite(f[touched]).any()
    np.testing.assert_array_equal(C[~touched], Co[~touched])
    np.testing.assert_allclose(f[~touched], sig[~touched], rtol=RTOL, atol=2.0 ** -40 / T)
