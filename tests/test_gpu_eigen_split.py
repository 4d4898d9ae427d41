"""Eigenpairs of 3x3 Cauchy-Green tensors of chosen spectra: spread over 12 orders of magnitude, nearly
aligned with the axes, nearly equal in pairs, equal, and tiny or huge as a whole.  Bounds from FP64
rounding: with u = 2^-53 and products of three terms, residuals and eigenvalues stay within 40 u lambda_max,
orthonormality within 40 u."""
import numpy as np
import pytest
import torch

from paper_2209_13775_gb300 import lcs

pytestmark = pytest.mark.gpu
BOUND = 40 * 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


def spectra(kind, m, rng):
    lam = 10.0 ** rng.uniform({"mild": -1, "wide": -12, "aligned": -10}.get(kind, -3), 0, (m, 3))
    if kind == "pairs":
        lam[:, 1] = lam[:, 0] * (1 - 10.0 ** rng.uniform(-13, -2, m))
    if kind == "equal":
        lam[:, 1] = lam[:, 0]
        lam[::2, 2] = lam[::2, 0]
    if kind == "tiny":
        lam *= 1e-60
    if kind == "huge":
        lam *= 1e60
    q = rng.standard_normal((m, 3, 3))
    if kind == "aligned":
        q = np.eye(3) + 1e-3 * q
    return lam, np.linalg.qr(q)[0]


@pytest.mark.parametrize("kind", ["mild", "wide", "aligned", "pairs", "equal", "tiny", "huge"])
def test_chosen_spectra(ctx, kind):
    m = 3000
    rng = np.random.default_rng(len(kind))
    lam, Q = spectra(kind, m, rng)
    G = np.sqrt(lam)[:, :, None] * np.swapaxes(Q, 1, 2)
    # central differences over a lattice of spacing 1 give G at disjoint centres (48 bits of it)
    n = (4 * m, 3, 3)
    x = np.zeros((3, n[0] * 9), np.float32)
    centre = 1 + 4 * np.arange(m) + n[0] * (1 + n[1])
    for b, st in enumerate((1, n[0], n[0] * n[1])):
        for a in range(3):
            p = (2 * G[:, a, b]).astype(np.float32)
            x[a, centre + st] = p
            x[a, centre - st] = (p - 2 * G[:, a, b]).astype(np.float32)
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
    ev, V = ev[centre].astype(np.longdouble), V[centre].astype(np.longdouble)
    top = ev[:, 2:]
    assert np.all(np.diff(ev, axis=1) >= 0) and np.all(top > 0)
    res = np.einsum("nij,nkj->nki", M, V) - ev[:, :, None] * V
    assert np.abs(res / top[:, :, None]).max() <= BOUND
    assert np.abs(np.einsum("nij,nkj->nik", V, V) - np.eye(3)).max() <= BOUND
    assert np.abs((ev.sum(1) - np.trace(M, axis1=1, axis2=2)) / top[:, 0]).max() <= BOUND
    assert np.all(np.take_along_axis(V, np.abs(V).argmax(2)[:, :, None], 2) > 0)
