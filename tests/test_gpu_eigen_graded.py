"""Eigenvalues of graded 3x3 Cauchy-Green tensors C = D S D, S well conditioned with a diagonal near 1 and D spanning
up to 17 orders of magnitude: the small eigenvalues carry a relative error, not one of the largest eigenvalue's.
Bound from FP64 rounding: rotations perturb C relatively and entry by entry, so with u = 2^-53 and k the condition
number of C scaled to a unit diagonal (Demmel and Veselic 1992) every eigenvalue is within 20 u k, relatively."""
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


def eigvals_long(M):
    """Jacobi rotations in extended precision (longdouble), ascending."""
    A = M.copy()
    for _ in range(12):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            r = 3 - p - q
            apq = A[:, p, q].copy()
            safe = np.where(apq == 0, 1, apq)
            tau = (A[:, q, q] - A[:, p, p]) / (2 * safe)
            t = np.where(apq == 0, 0, np.where(tau < 0, -1, 1) / (np.abs(tau) + np.hypot(tau, np.longdouble(1))))
            c = 1 / np.sqrt(t * t + 1)
            s = t * c
            A[:, p, p] -= t * apq
            A[:, q, q] += t * apq
            x, y = A[:, r, p].copy(), A[:, r, q].copy()
            A[:, p, q] = A[:, q, p] = 0
            A[:, r, p] = A[:, p, r] = c * x - s * y
            A[:, r, q] = A[:, q, r] = s * x + c * y
    return np.sort(np.einsum("nii->ni", A), axis=1)


@pytest.mark.parametrize("kind,span", [("step", 6), ("step", 11), ("step", 13), ("step", 15), ("step", 17), ("two", 13),
                                       ("two", 15), ("one", 15), ("one", 17)])
def test_graded(ctx, kind, span):
    m = 2000
    rng = np.random.default_rng(span)
    D = np.array({"step": (1.0, 10.0 ** (-span / 2), 10.0 ** -span), "two": (1.0, 10.0 ** -span, 10.0 ** -span),
                  "one": (1.0, 1.0, 10.0 ** -span)}[kind])
    G = np.eye(3) + rng.uniform(-0.4, 0.4, (m, 3, 3))
    for i in range(m):
        G[i] *= rng.permutation(D)          # columns: C = G^T G is graded on both sides
    n = (4 * m, 3, 3)
    x = np.zeros((3, n[0] * 9), np.float32)
    centre = 1 + 4 * np.arange(m) + n[0] * (1 + n[1])
    for b, st in enumerate((1, n[0], n[0] * n[1])):
        for a in range(3):
            x[a, centre + st] = G[:, a, b]
            x[a, centre - st] = -G[:, a, b]
    seeds = lcs.lcs_seed_grid(ctx, lcs.seed_desc(3, n, (0.0,) * 3, (n[0] - 1.0, 2.0, 2.0)))
    N = lcs.lcs_seeds_count(seeds)
    fm = lcs.lcs_flowmap_create(ctx, seeds, 1)
    C, ev, V = np.empty((N, 6)), np.empty((N, 3)), np.empty((N, 3, 3))
    try:
        lcs.lcs_flowmap_set(ctx, fm, 0, x, np.zeros(N, np.uint8), 1.0)
        lcs.lcs_cauchy_green(ctx, fm, 0, C)
        lcs.lcs_cg_eigen(ctx, fm, 0, ev, V)
    finally:
        lcs.lcs_free_flowmap(fm)
        lcs.lcs_free_seeds(seeds)
    a, b, c, d, e, f = C[centre].astype(np.longdouble).T
    M = np.stack([np.stack([a, b, c], -1), np.stack([b, d, e], -1), np.stack([c, e, f], -1)], -2)
    s = np.sqrt(np.einsum("nii->ni", M))
    k = np.linalg.cond((M / s[:, :, None] / s[:, None, :]).astype(np.float64))
    assert k.max() < 1e6
    ref = eigvals_long(M)
    err = np.abs(ev[centre] / ref - 1).astype(np.float64) / k[:, None]
    assert err.max() <= 20 * 2.0 ** -53, err.max(0) * 2.0 ** 53
    assert np.abs(np.einsum("nij,nkj->nik", V[centre], V[centre]) - np.eye(3)).max() <= 40 * 2.0 ** -53
