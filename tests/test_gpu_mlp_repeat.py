"""Gradients of the learned proposal's network repeat bitwise where their sums have a fixed order: all of them for batches
below 512 samples (one writer an entry), the bias gradients for every batch."""
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
