"""The tiled FP32 element products of meshes without hex patches (linear tets in an order with locality) and of
quadratic tets, against the oracle's matrices: case counts 4 to 32, a ragged last tile, elements without locality
(no tiles: the element kernel), Dirichlet rows, and infinities and NaN, which have to reach exactly the rows of
their elements.  Bounds as in the other FP32 product tests: 2e-6 (linear) and 5e-6 (quadratic) of the largest entry."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from oracle import tet10_oracle
from paper_2409_20380_gb300 import build, fem
from paper_2409_20380_gb300 import workload as wl
from helpers import small_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_dev():
    import torch
    build.build()
    fem.lib()
    return torch


TP = wl.TimeParams()
CM, CK = 4.0 / TP.dt ** 2 + 2.0 * TP.a0 / TP.dt, 1.0 + 2.0 * TP.a1 / TP.dt


def _tets(local):
    # 79,488 tets and 5 fewer: 311 tiles of 256, the last one ragged
    m = small_mesh(24, 23, 24, h=1.0 / 16, perturb=0.1)
    rng = np.random.default_rng(5)
    order = np.argsort(np.arange(m.n_elems) + (rng.uniform(0, 96, m.n_elems) if local else rng.uniform(0, 1e7, m.n_elems)))[5:]
    m.conn, m.mat_id = np.ascontiguousarray(m.conn[order]), np.ascontiguousarray(m.mat_id[order])
    return m


def _csr(conn, K, M, n, fixed):
    npe = conn.shape[1]
    dof = (3 * conn[:, :, None].astype(np.int64) + np.arange(3)).reshape(-1, 3 * npe)
    A = sp.csr_matrix(((CM * M + CK * K).reshape(-1), (np.repeat(dof, 3 * npe, axis=1).reshape(-1),
                                                        np.tile(dof, (1, 3 * npe)).reshape(-1))), shape=(3 * n, 3 * n))
    free = sp.diags((fixed == 0).astype(float))
    return free @ A


def _apply(torch, f, h, p, r, ptq=None):
    d = torch.tensor(p.reshape(-1), dtype=torch.float32, device="cuda")
    q = torch.full_like(d, float("nan"))
    if ptq is None:
        f(h, d, q, r, CM, CK)
    else:
        f(h, d, q, r, CM, CK, ptq)
    return q.cpu().numpy().astype(np.float64).reshape(p.shape)


def _check(torch, f, h, A, n, fixed, r, tol, ptq_too):
    rng = np.random.default_rng(r)
    p = (rng.standard_normal((3 * n, r)) * (fixed == 0)[:, None]).astype(np.float32)
    p[:, 0] *= 1e-30          # cases of very different size share the tiles
    p[:, r - 1] *= 1e20
    ref = A @ p.astype(np.float64)
    ptq = torch.empty(r, dtype=torch.float64, device="cuda")
    for red in ([None, ptq] if ptq_too else [None]):
        q = _apply(torch, f, h, p, r, red)
        assert np.all(np.abs(q - ref).max(axis=0) <= tol * np.abs(ref).max(axis=0))
        assert np.all(q[fixed == 1] == 0.0)
        if red is not None:
            want = (p.astype(np.float64) * ref).sum(axis=0)
            got = ptq.cpu().numpy()
            mid = slice(1, r - 1)     # (the FP32 products p q of the two scaled cases leave FP32's range)
            assert np.all(np.abs(got - want)[mid] <= tol * np.abs(want)[mid])
    # an infinity and a NaN in two cases: non-finite exactly in the rows their columns touch
    bad = p.copy()
    free_dofs = np.nonzero(fixed == 0)[0]
    i, j = free_dofs[len(free_dofs) // 3], free_dofs[len(free_dofs) // 2]
    bad[i, 1], bad[j, 2] = np.inf, np.nan
    q = _apply(torch, f, h, bad, r)
    pattern = (abs(A) > 0).astype(np.float64)
    for c, d in ((1, i), (2, j)):
        hit = np.asarray(pattern[:, d].todense()).reshape(-1) > 0
        got = ~np.isfinite(q[:, c])
        assert np.all(got[hit]), c
        # (an element's other rows may turn non-finite through 0 * inf; never a row of no shared element)
        node_hit = np.repeat(hit.reshape(-1, 3).any(axis=1), 3)
        assert not np.any(got[~node_hit]), c
        clean = ~node_hit
        assert np.all(np.abs(q[clean, c] - (A @ np.where(np.isfinite(bad), bad, 0).astype(np.float64))[clean, c])
                      <= 10 * tol * np.abs(ref[:, c]).max())


@pytest.mark.parametrize("local", [True, False])
def test_linear_tets(torch_dev, local):
    m = _tets(local)
    K, M = oracle.tet4_element_matrices(m.xyz, m.conn, m.mat_id, m.lam_mu_rho)
    A = _csr(m.conn, K, M, m.n_nodes, m.fixed_dof)
    h = fem.fem_mesh_create(m, TP)
    try:
        for r in (4, 8, 16, 32) if local else (8,):
            _check(torch_dev, fem.fem_ebe_apply, h, A, m.n_nodes, m.fixed_dof, r, 2e-6, False)
    finally:
        fem.fem_mesh_destroy(h)


def test_quadratic_tets(torch_dev):
    m4 = small_mesh(17, 17, 17, h=1.0 / 16, perturb=0.1)      # 29,478 elements: 308 tiles of 96, the last ragged
    m = wl.tet10_mesh_ordered(m4)[0]
    K, M = tet10_oracle.tet10_element_matrices(m.xyz, m.conn, m.mat_id, m.lam_mu_rho)
    A = _csr(m.conn, K, M, m.n_nodes, m.fixed_dof)
    h = fem.fem_mesh10_create(m)
    try:
        for r in (1, 4, 16, 32):
            if r == 1:
                p = (np.random.default_rng(0).standard_normal((3 * m.n_nodes, 1)) * (m.fixed_dof == 0)[:, None])
                ref = A @ p.astype(np.float32).astype(np.float64)
                q = _apply(torch_dev, fem.fem_ebe10_apply, h, p, 1)
                assert np.abs(q - ref).max() <= 5e-6 * np.abs(ref).max()
            else:
                _check(torch_dev, fem.fem_ebe10_apply, h, A, m.n_nodes, m.fixed_dof, r, 5e-6, True)
    finally:
        fem.fem_mesh10_destroy(h)
