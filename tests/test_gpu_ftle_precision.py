"""FTLE where the eigenvalue's own error would show in it: lambda_max within 1e-7 to 1e-2 of 1, the two largest
eigenvalues apart, 1e-1 to 1e-7 from each other, or equal, in random orientations.  sigma = ln(lambda) / (2 |T|) against
FP64 eigenvalues of the library's C (bit-identical to the plain FP64 definition): the logarithm and two products
round within 3 ulps of 2^-23; lambda's error is 2^-46 where it comes from FP64 (the cubic's root), and where it does
not at most 2^-30 of the logarithm."""
import numpy as np
import pytest
import torch

from paper_2209_13775_gb300 import lcs

pytestmark = pytest.mark.gpu
T = 1.25
M = 4000


@pytest.mark.parametrize("pair", ["apart", "near", "equal"])
@pytest.mark.parametrize("dim", [2, 3])
def test_sigma_near_zero(dim, pair):
    torch.cuda.set_device(0)
    ctx = lcs.lcs_create(0, torch.cuda.current_stream())
    rng = np.random.default_rng(10 * dim + len(pair))
    lam = np.empty((M, dim))
    lam[:, 0] = 1 + rng.choice([-1, 1], M) * 10.0 ** rng.uniform(-7, -2, M)
    gap = {"apart": rng.uniform(0.2, 0.9, M), "near": 10.0 ** rng.uniform(-7, -1, M), "equal": np.zeros(M)}[pair]
    lam[:, 1] = lam[:, 0] * (1 - gap)
    if dim == 3:
        lam[:, 2] = lam[:, 1] * 10.0 ** rng.uniform(-4, -0.3, M)
    Q = np.linalg.qr(rng.standard_normal((M, dim, dim)))[0]
    G = np.sqrt(lam)[:, :, None] * np.swapaxes(Q, 1, 2)
    # central differences over a lattice of spacing 1 give G at disjoint centres (48 bits of it)
    n = (4 * M, 3, 3)[:dim]
    x = np.zeros((dim, int(np.prod(n))), np.float32)
    strides = (1, n[0], n[0] * n[1])[:dim]
    centre = 1 + 4 * np.arange(M) + sum(strides[1:])
    for b, st in enumerate(strides):
        for a in range(dim):
            p = (2 * G[:, a, b]).astype(np.float32)
            x[a, centre + st] = p
            x[a, centre - st] = (p - 2 * G[:, a, b]).astype(np.float32)
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(dim, n, (0.0,) * dim, tuple(v - 1.0 for v in n)))
    N = lcs.lcs_seeds_count(seeds)
    fm = lcs.lcs_flowmap_create(ctx, seeds, 1)
    f, f2, C = np.empty(N, np.float32), np.empty(N, np.float32), np.empty((N, dim * (dim + 1) // 2))
    try:
        lcs.lcs_flowmap_set(ctx, fm, 0, x, np.zeros(N, np.uint8), T)
        lcs.lcs_ftle(ctx, fm, 0, f)
        lcs.lcs_ftle(ctx, fm, 0, f2, None, C)
    finally:
        lcs.lcs_free_flowmap(fm)
        lcs.lcs_free_seeds(seeds)
        lcs.lcs_destroy(ctx)
    np.testing.assert_array_equal(f, f2)
    S = np.empty((M, dim, dim))
    for q, (i, j) in enumerate(zip(*np.triu_indices(dim))):
        S[:, i, j] = S[:, j, i] = C[centre, q]
    lm = np.linalg.eigvalsh(S)[:, -1]
    sig = np.log1p(lm - 1) / (2 * T)
    np.testing.assert_allclose(f[centre], sig, rtol=3 * 2.0 ** -23 + 2.0 ** -30, atol=2.0 ** -46 / (2 * T))
