"""The fused training step at the edges of its 96-sample tiles and of one tile per CTA, against the FP64
oracle on the same BF16 weights, with the tolerances of the network tests (relative L2 2e-2 and cosine 0.999
per tensor, loss 1e-2: BF16 activations); repeated calls give the same bits; an Adam step leaves the operand
tiles that a network made from the new parameters has."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2209_13775_gb300 import inputs, lcs
from test_gpu_mlp import GYRE_FEAT, bf16_params, cosine, mlp_handle, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


@pytest.mark.parametrize("n", [128, 384, 14592, 14720, 29184, 29312])
def test_gradients_at_tile_edges(ctx, n):
    p = inputs.mlp_init(seed=200 + n)
    rng = np.random.default_rng(n)
    for o in (896, 17408, 33920, 50432):   # biases that are not zero
        p[o:o + 128] = rng.normal(scale=0.1, size=128).astype(np.float32)
    p[-3:] = [0.05, -0.02, -2.0]
    m = mlp_handle(ctx, p)
    xyt = inputs.surrogate_samples(n, seed=201 + n)
    disp = rng.normal(scale=0.05, size=(2, n)).astype(np.float32)
    g, g2 = (np.empty(omlp.NPARAMS, dtype=np.float32) for _ in range(2))
    loss = lcs.lcs_mlp_loss_grad(ctx, m, xyt, disp, 0.25, g)
    assert lcs.lcs_mlp_loss_grad(ctx, m, xyt, disp, 0.25, g2) == loss
    np.testing.assert_array_equal(g, g2)
    phi = omlp.features(*(xyt[k].astype(np.float64) for k in range(3)), **GYRE_FEAT)
    lo, go = omlp.loss_and_grad(bf16_params(p), phi, disp.astype(np.float64), 0.1, 0.25)
    assert abs(loss - lo) <= 1e-2 * abs(lo)
    o = 0
    for i, s in enumerate(omlp.SHAPES):
        k = int(np.prod(s))
        a, b = g[o:o + k].astype(np.float64), go[o:o + k]
        assert rel_err(a, b) <= 2e-2 and cosine(a, b) >= 0.999, (i, rel_err(a, b), cosine(a, b))
        o += k
    lcs.lcs_mlp_adam(ctx, m, lr=1e-2)
    q = np.empty(omlp.NPARAMS, dtype=np.float32)
    lcs.lcs_mlp_get_params(ctx, m, q)
    assert not np.array_equal(p, q)
    fresh = mlp_handle(ctx, q)
    out = [np.empty((3, 128), dtype=np.float32) for _ in range(2)]
    for h, y in zip((m, fresh), out):
        lcs.lcs_mlp_forward(ctx, h, np.ascontiguousarray(xyt[:, :128]), y)
        lcs.lcs_mlp_free(h)
    np.testing.assert_array_equal(*out)
