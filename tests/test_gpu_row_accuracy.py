"""Every row of the FP32 products of meshes without hex patches and of quadratic tets keeps FP32's accuracy relative to
its own terms, |A| |p|, on meshes whose rows and values differ by many orders of magnitude between neighbours: a layer
10,000 times stiffer than its neighbour, elements whose edges grow 8 : 1, values that fall off by eight decades,
negative lambda.

Bound: 2e-6 of the row's sum of |a_ij| |p_j| over its elements: a contribution of a few rounded operations and a sum of
up to 60 of them, 32 units of 2^-24."""
import numpy as np
import pytest

import oracle
from oracle import tet10_oracle
from paper_2409_20380_gb300 import build, fem
from paper_2409_20380_gb300 import workload as wl
from helpers import small_mesh
from test_gpu_elem_tile import CK, CM, TP, _csr, _tets

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_dev():
    import torch
    build.build()
    fem.lib()
    return torch


def _uneven(m, kind):
    m.lam_mu_rho = m.lam_mu_rho.copy()
    if "contrast" in kind:
        m.lam_mu_rho[0, :2] *= 1e4
    if "graded" in kind:
        m.xyz[:] *= (2.0 ** (3.0 * m.xyz[:, 2] / m.xyz[:, 2].max()))[:, None]
    if "auxetic" in kind:
        m.lam_mu_rho[:, 0] = -0.6 * m.lam_mu_rho[:, 1]
    return m


def _check(torch, f, h, m, K, M, r, kind):
    n = m.n_nodes
    A = _csr(m.conn, K, M, n, m.fixed_dof)
    absA = _csr(m.conn, np.abs(CM * M + CK * K) / CK, np.zeros_like(M), n, m.fixed_dof)
    rng = np.random.default_rng(r)
    p = rng.standard_normal((3 * n, r)) * (m.fixed_dof == 0)[:, None]
    if "decay" in kind:
        d = np.linalg.norm(m.xyz - m.xyz[n // 2], axis=1)
        p *= np.repeat(10.0 ** (-8.0 * d / d.max()), 3)[:, None]
    p = p.astype(np.float32)
    ref, bound = A @ p.astype(np.float64), absA @ np.abs(p.astype(np.float64))
    x = torch.tensor(p.reshape(-1), device="cuda")
    for red in (None, torch.empty(r, dtype=torch.float64, device="cuda")):
        q = torch.full_like(x, float("nan"))
        f(h, x, q, r, CM, CK, red)
        err = np.abs(q.cpu().numpy().astype(np.float64).reshape(p.shape) - ref)
        assert np.all(err <= 2e-6 * bound), (float((err[bound > 0] / bound[bound > 0]).max()), red is not None)


KINDS = ["contrast", "graded", "decay", "contrast graded decay", "auxetic"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("r", [4, 8])
def test_linear_tets(torch_dev, kind, r):
    m = _uneven(_tets(True), kind)
    K, M = oracle.tet4_element_matrices(m.xyz, m.conn, m.mat_id, m.lam_mu_rho)
    h = fem.fem_mesh_create(m, TP)
    try:
        _check(torch_dev, fem.fem_ebe_apply, h, m, K, M, r, kind)
    finally:
        fem.fem_mesh_destroy(h)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("r", [8, 16])
def test_quadratic_tets(torch_dev, kind, r):
    m = wl.tet10_mesh_ordered(_uneven(small_mesh(14, 14, 14, h=1.0 / 16, perturb=0.1), kind))[0] 
    K, M = tet10_oracle.tet10_element_matrices(m.xyz, m.conn, m.mat_id, m.lam_mu_rho)
    h = fem.fem_mesh10_create(m)
    try:
        _check(torch_dev, fem.fem_ebe10_apply, h, m, K, M, r, kind)
    finally:
        fem.fem_mesh10_destroy(h)
