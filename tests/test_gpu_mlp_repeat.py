"""Gradients of the learned proposal's network repeat bitwise where their sums have a fixed order: all of them for batches
below 512 samples (one writer an entry), the bias gradients for every batch.  Results may be written over the inputs."""
import numpy as np
import pytest

from paper_2409_20380_gb300 import build, fem
from paper_2409_20380_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_dev():
    import torch
    build.build()
    fem.lib()
    return torch


@pytest.mark.parametrize("B", [33, 100, 300, 511, 4096])
@pytest.mark.parametrize("residual", [False, True])
def test_gradient_repeats(torch_dev, B, residual):
    torch = torch_dev
    rng = np.random.default_rng(B)
    x = torch.tensor(rng.standard_normal((B, 64)).astype(np.float32), device="cuda")
    t = torch.tensor(rng.standard_normal((B, fem.FEM_MLP_RES if residual else 32)).astype(np.float32), device="cuda")
    biases = torch.zeros(fem.FEM_MLP_N_PARAMS, dtype=torch.bool, device="cuda")
    o = 0
    for n_in, n_out in ((64, 256), (256, 256), (256, 32)):
        o += n_in * n_out + n_out
        biases[o - n_out:o] = True
    net = fem.fem_mlp_create(wl.mlp_init_weights(5).astype(np.float32))
    f = fem.fem_mlp_loss_grad_residual if residual else fem.fem_mlp_loss_grad
    try:
        first = None
        for _ in range(20):
            g = torch.full((fem.FEM_MLP_N_PARAMS,), float("nan"), device="cuda")
            f(net, x, t, g)
            assert bool(torch.isfinite(g).all())
            if first is None:
                first = g
            assert torch.equal(g[biases], first[biases])
            assert B >= 512 or torch.equal(g, first)
    finally:
        fem.fem_mlp_destroy(net)


def test_results_over_inputs(torch_dev):
    torch = torch_dev
    B = 40000      # more blocks than run at once
    rng = np.random.default_rng(1)
    x = torch.tensor(rng.standard_normal((B, 64)).astype(np.float32), device="cuda")
    t = torch.tensor(rng.standard_normal((B, 32)).astype(np.float32), device="cuda")
    net = fem.fem_mlp_create(wl.mlp_init_weights(5).astype(np.float32))
    try:
        out, g = torch.empty((B, 32), device="cuda"), torch.empty(fem.FEM_MLP_N_PARAMS, device="cuda")
        fem.fem_mlp_forward(net, x, out)
        loss = fem.fem_mlp_loss_grad(net, x, t, g)
        both = torch.empty(96 * B, device="cuda")     # x, then t
        for over in (0, 1000, 64 * B - 90000, 64 * B - 16, 64 * B):
            both[:64 * B], both[64 * B:] = x.reshape(-1), t.reshape(-1)
            y = both[over:over + 32 * B]
            fem.fem_mlp_forward(net, both[:64 * B].reshape(B, 64), y.reshape(B, 32))
            assert torch.equal(y.reshape(B, 32), out), over
            both[:64 * B], both[64 * B:] = x.reshape(-1), t.reshape(-1)
            y = both[over:over + fem.FEM_MLP_N_PARAMS]
            got = fem.fem_mlp_loss_grad(net, both[:64 * B].reshape(B, 64), both[64 * B:].reshape(B, 32), y)
            assert abs(got - loss) <= 1e-12 * abs(loss)
            assert float((y - g).abs().max()) <= 1e-6 * float(g.abs().max()), over   # (the order of 13 atomic adds)
    finally:
        fem.fem_mlp_destroy(net)
