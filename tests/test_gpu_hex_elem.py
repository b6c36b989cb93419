"""The kernels that fem_ebe_apply chooses by itself on hex patches for FP32 products of one or two cases and for FP64
products: as exact as the tiled ones (whose corner sums over a hex's tets stay in registers), Dirichlet rows zero, sizes
at the edges of the choice (H r = 11,000) and of a block.

The rms error against wider arithmetic, a mean over 20 vectors (its own spread is below 1%), is at most 6% above the
tiles'; one atomic add a tet instead of a hex is 10% to 45% above.  The reference of FP64 products is summed in
numpy's long double."""
import numpy as np
import pytest

from paper_2409_20380_gb300 import build, fem
from paper_2409_20380_gb300 import workload as wl
from helpers import small_mesh

pytestmark = pytest.mark.gpu
TP = wl.TimeParams()
CM, CK = 4.0 / TP.dt ** 2 + 2.0 * TP.a0 / TP.dt, 1.0 + 2.0 * TP.a1 / TP.dt


@pytest.fixture(scope="module")
def torch_dev():
    import torch
    build.build()
    fem.lib()
    return torch


def _operator(m, dtype, cM=CM, cK=CK):
    """p -> (cM M + cK K) p from the tets' gradients, in long double for FP64 products."""
    wide = np.longdouble if dtype == "float64" else np.float64
    x = m.xyz.astype(wide)[m.conn]
    e = [x[:, i] - x[:, 0] for i in (1, 2, 3)]
    det = (e[0] * np.cross(e[1], e[2])).sum(axis=1)
    g = np.stack([np.cross(e[1], e[2]), np.cross(e[2], e[0]), np.cross(e[0], e[1])], axis=1) / det[:, None, None]
    g = np.concatenate([-g.sum(axis=1, keepdims=True), g], axis=1)
    lam, mu, rho = (m.lam_mu_rho.astype(wide)[m.mat_id].T * (det / 6))[:, :, None, None, None]
    free = (m.fixed_dof == 0)

    def apply(p):
        u = p.astype(wide).reshape(m.n_nodes, 3, -1)[m.conn]                      # [e][a][i][case]
        G = np.einsum("eaj,eaic->eijc", g, u)
        S = mu * (G + G.transpose(0, 2, 1, 3))
        tr = lam[:, 0, 0] * (G[:, 0, 0] + G[:, 1, 1] + G[:, 2, 2])
        for i in range(3):
            S[:, i, i] += tr
        f = cK * np.einsum("eaj,eijc->eaic", g, S) + cM * rho / 20 * (u + u.sum(axis=1, keepdims=True))
        q = np.zeros((m.n_nodes, 3, f.shape[3]), dtype=wide)
        np.add.at(q, m.conn.reshape(-1), f.reshape((-1,) + f.shape[2:]))
        return q.reshape(p.shape) * free[:, None]

    return apply


@pytest.mark.parametrize("dtype,dims,r", [("float32", (8, 8, 8), 1), ("float32", (12, 11, 10), 2), ("float64", (8, 8, 8), 1),
                                          ("float64", (9, 8, 7), 4), ("float64", (12, 12, 10), 8)])
def test_as_exact_as_tiles(torch_dev, dtype, dims, r):
    torch = torch_dev
    m, tp = wl.config2_mesh(*dims), wl.config2_time_params()
    cM, cK = 4.0 / tp.dt ** 2 + 2.0 * tp.a0 / tp.dt, 1.0 + 2.0 * tp.a1 / tp.dt
    apply = _operator(m, dtype, cM, cK)
    h = fem.fem_mesh_create(m, tp)
    try:
        rms = {0: [], 2: []}
        for seed in range(20 if r < 8 else 6):
            p = np.random.default_rng(seed).standard_normal((3 * m.n_nodes, r)) * (m.fixed_dof == 0)[:, None]
            x = torch.tensor(p.reshape(-1), dtype=getattr(torch, dtype), device="cuda")
            ref = apply(x.cpu().numpy().reshape(p.shape))
            for variant in (0, 2):
                fem.fem_mesh_tune(h, variant, 0)
                q = torch.full_like(x, float("nan"))
                fem.fem_ebe_apply(h, x, q, r, cM, cK)
                err = q.cpu().numpy().reshape(p.shape) - ref
                rms[variant].append(float(np.sqrt((err ** 2).mean() / (ref ** 2).mean())))
        assert np.mean(rms[0]) <= 1.06 * np.mean(rms[2]), rms
    finally:
        fem.fem_mesh_destroy(h)


# hexes x cases at and above 11,000, one hex, blocks with a remainder
@pytest.mark.parametrize("dtype,dims,r", [("float64", (1, 1, 1), 1), ("float64", (1, 1, 1), 32), ("float64", (3, 2, 5), 2),
                                          ("float64", (7, 3, 3), 4), ("float64", (8, 8, 8), 16), ("float64", (9, 9, 7), 16),
                                          ("float64", (11, 10, 25), 4), ("float64", (11, 10, 26), 4), ("float64", (8, 8, 4), 32),
                                          ("float32", (1, 1, 1), 2), ("float32", (27, 27, 27), 2), ("float32", (28, 27, 27), 2)])
def test_edges(torch_dev, dtype, dims, r):
    torch = torch_dev
    m = small_mesh(*dims)
    apply = _operator(m, "float32")
    tol = 1e-13 if dtype == "float64" else 2e-6
    p = np.random.default_rng(r).standard_normal((3 * m.n_nodes, r)) * (m.fixed_dof == 0)[:, None]
    x = torch.tensor(p.reshape(-1), dtype=getattr(torch, dtype), device="cuda")
    p = x.cpu().numpy().reshape(p.shape).astype(np.float64)
    ref = apply(p)
    h = fem.fem_mesh_create(m, TP)
    try:
        for ptq in (None, torch.empty(r, dtype=torch.float64, device="cuda")):
            q = torch.full_like(x, float("nan"))
            fem.fem_ebe_apply(h, x, q, r, CM, CK, ptq)
            got = q.cpu().numpy().reshape(p.shape).astype(np.float64)
            assert np.all(np.abs(got - ref).max(axis=0) <= tol * np.abs(ref).max(axis=0))
            assert np.all(got[m.fixed_dof == 1] == 0.0)
            if ptq is not None:
                want = (p * ref).sum(axis=0)
                assert np.all(np.abs(ptq.cpu().numpy() - want) <= tol * np.abs(want))
    finally:
        fem.fem_mesh_destroy(h)
