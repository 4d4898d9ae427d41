"""A block of the network's kernels that gives up its wait for the weights: with a limit under a microsecond it tests
their copy once, right behind the launch of the copy (107 KB), which no block finds complete.  It waits for the copy
all the same before it exits, lcs_synchronize reports LCS_ETIMEOUT, and with the default limit the same network then
gives the same results as before.  Nothing traps or spins without bound."""
import numpy as np
import pytest
import torch

from paper_2209_13775_gb300 import inputs, lcs
from test_gpu_mlp import mlp_handle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = lcs.lcs_create(0, torch.cuda.current_stream())
    yield c
    lcs.lcs_destroy(c)


def device_inputs(n, seed):
    xyt = torch.from_numpy(inputs.surrogate_samples(n, seed=seed)).cuda()
    disp = torch.from_numpy(np.random.default_rng(seed).normal(scale=0.05, size=(2, n)).astype(np.float32)).cuda()
    return xyt, disp


def timed_out(ctx):
    try:
        lcs.lcs_synchronize(ctx)
    except lcs.LcsError as e:
        return e.status == 4          # LCS_ETIMEOUT
    return False


@pytest.mark.parametrize("n", [128, 4096, 65536])
def test_forward(ctx, n):
    m = mlp_handle(ctx, inputs.mlp_init(seed=n))
    xyt, _ = device_inputs(n, n)
    out = [torch.empty(3, n, device="cuda") for _ in range(2)]
    try:
        lcs.lcs_mlp_forward(ctx, m, xyt, out[0])
        lcs.lcs_synchronize(ctx)
        lcs.lcs_mlp_set_wait_limit(ctx, m, 1e-9)
        lcs.lcs_mlp_forward(ctx, m, xyt, out[1])
        assert timed_out(ctx)
        lcs.lcs_mlp_set_wait_limit(ctx, m, 0.0)
        lcs.lcs_mlp_forward(ctx, m, xyt, out[1])
        lcs.lcs_synchronize(ctx)
        assert torch.equal(*out)
        for bad in (-1.0, 61.0, float("nan")):
            with pytest.raises(lcs.LcsError) as e:
                lcs.lcs_mlp_set_wait_limit(ctx, m, bad)
            assert e.value.status == 1
    finally:
        lcs.lcs_mlp_free(m)


@pytest.mark.parametrize("n", [128, 4096, 65536])
def test_loss_grad(ctx, n):
    m = mlp_handle(ctx, inputs.mlp_init(seed=n))
    xyt, disp = device_inputs(n, n)
    g = [torch.empty(lcs.MLP_NPARAMS, device="cuda") for _ in range(2)]
    try:
        loss = lcs.lcs_mlp_loss_grad(ctx, m, xyt, disp, 0.25, g[0])
        lcs.lcs_synchronize(ctx)
        lcs.lcs_mlp_set_wait_limit(ctx, m, 1e-9)
        assert np.isnan(lcs.lcs_mlp_loss_grad(ctx, m, xyt, disp, 0.25, g[1]))
        assert timed_out(ctx)
        assert not g[1].any()         # no block had its weights: nothing, and nothing of the batch before
        lcs.lcs_mlp_set_wait_limit(ctx, m, 0.0)
        assert lcs.lcs_mlp_loss_grad(ctx, m, xyt, disp, 0.25, g[1]) == loss
        lcs.lcs_synchronize(ctx)
        assert torch.equal(*g)
    finally:
        lcs.lcs_mlp_free(m)
