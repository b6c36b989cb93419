"""The inner solves' passes with two cases a thread (from 450,000 threads' work on: 8 cases on 112,500 to 225,000 nodes, 2
cases on 450,000): every case takes the iterations it takes with one case a thread, within 2 (one an inner solve: the order of the sums), and
its residual, by the FP64 product, is below the tolerance."""
import pytest

from paper_2409_20380_gb300 import build, fem
from paper_2409_20380_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,r,few", [((60, 55, 35), 8, 4), ((80, 80, 70), 2, 1)])
def test_same_iterations(dims, r, few):
    import torch
    build.build()
    m, tp = wl.config2_mesh(*dims), wl.config2_time_params()
    cM, cK = 4.0 / tp.dt ** 2 + 2.0 * tp.a0 / tp.dt, 1.0 + 2.0 * tp.a1 / tp.dt
    free = torch.tensor((m.fixed_dof == 0).astype(float), device="cuda")
    b = torch.randn((3 * m.n_nodes, r), generator=torch.Generator(device="cuda").manual_seed(3), dtype=torch.float64,
                    device="cuda") * free[:, None]
    b[:, r - 1] *= 1e-6          # (cases of different size converge on their own)
    opts = fem.fem_opts_default(precision=fem.FEM_FP32_INNER, tol=1e-9)
    h = fem.fem_mesh_create(m, tp)
    try:
        def solve(cols):
            rhs = b[:, cols].contiguous()
            x = torch.zeros_like(rhs)
            iters = fem.pcg_solve(h, rhs, x, len(cols), opts)[1]
            q = torch.empty_like(x)
            fem.fem_ebe_apply(h, x, q, len(cols), cM, cK)
            res = (rhs - q).norm(dim=0) / rhs.norm(dim=0)
            assert bool((res <= 1.001e-9).all()), res
            return list(iters)

        all_cols = list(range(r))
        pairs = solve(all_cols)
        alone = [i for k in range(0, r, few) for i in solve(all_cols[k:k + few])]
        assert all(abs(p - a) <= 2 for p, a in zip(pairs, alone)), (pairs, alone)
    finally:
        fem.fem_mesh_destroy(h)
