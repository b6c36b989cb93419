"""FP32 products of very small vectors, whose tile sums are fixed point: the scale in and the scale back have to cancel
down to FP32's smallest normal numbers.  Linear tets without hex patches, quadratic tets, and the hex kernels
(automatic, packed, FP16 matrices), with and without p^T q, M alone and A.

Bound: a row of at most 80 contributions, each rounded to 2^-127 at the least (FP32 atomics flush below 2^-126), so
80 x 2^-126, and the relative bound of the other tests of each kernel (2e-6 linear, 5e-6 quadratic, 2e-3 FP16)."""
import numpy as np
import pytest

import oracle
from oracle import tet10_oracle
from paper_2409_20380_gb300 import build, fem
from paper_2409_20380_gb300 import workload as wl
from helpers import small_mesh
from test_gpu_elem_tile import CK, CM, TP, _csr, _tets

pytestmark = pytest.mark.gpu
FLOOR = 80 * 2.0 ** -126
SCALES = [2.0 ** -70, 2.0 ** -86, 2.0 ** -90, 2.0 ** -94, 2.0 ** -98, 2.0 ** -102, 2.0 ** -110, 2.0 ** -118]


@pytest.fixture(scope="module")
def torch_dev():
    import torch
    build.build()
    fem.lib()
    return torch


def _check(torch, f, h, m, K, M, coeffs, r, tol):
    rng = np.random.default_rng(17)
    p = rng.standard_normal((3 * m.n_nodes, r)) * (m.fixed_dof == 0)[:, None]
    for a_m, a_k in coeffs:
        # (_csr takes CM M + CK K)
        A = _csr(m.conn, K * (a_k / CK), M * (a_m / CM), m.n_nodes, m.fixed_dof)
        for scale in SCALES:
            x = (p * scale).astype(np.float32)
            x[:, 0] = p[:, 0]        # a case of ordinary size beside the small ones
            ref = A @ x.astype(np.float64)
            d = torch.tensor(x.reshape(-1), device="cuda")
            for red in (None, torch.empty(r, dtype=torch.float64, device="cuda")):
                q = torch.full_like(d, float("nan"))
                f(h, d, q, r, a_m, a_k, red)
                err = np.abs(q.cpu().numpy().astype(np.float64).reshape(x.shape) - ref).max(axis=0)
                assert np.all(err <= tol * np.abs(ref).max(axis=0) + FLOOR), (a_m, a_k, scale, red is not None)


def test_linear_tets(torch_dev):
    m = _tets(True)
    K, M = oracle.tet4_element_matrices(m.xyz, m.conn, m.mat_id, m.lam_mu_rho)
    h = fem.fem_mesh_create(m, TP)
    try:
        _check(torch_dev, fem.fem_ebe_apply, h, m, K, M, ((1.0, 0.0), (0.0, 1.0), (CM, CK)), 8, 2e-6)
    finally:
        fem.fem_mesh_destroy(h)


def test_quadratic_tets(torch_dev):
    m = wl.tet10_mesh_ordered(small_mesh(17, 17, 17, h=1.0 / 16, perturb=0.1))[0]
    K, M = tet10_oracle.tet10_element_matrices(m.xyz, m.conn, m.mat_id, m.lam_mu_rho)
    h = fem.fem_mesh10_create(m)
    try:
        _check(torch_dev, fem.fem_ebe10_apply, h, m, K, M, ((1.0, 0.0), (CM, CK)), 8, 5e-6)
    finally:
        fem.fem_mesh10_destroy(h)


@pytest.mark.parametrize("variant", [0, 5, 6, 7, 9])
def test_hex_kernels(torch_dev, variant):
    m = small_mesh(12, 12, 12, h=1.0 / 16)
    K, M = oracle.tet4_element_matrices(m.xyz, m.conn, m.mat_id, m.lam_mu_rho)
    h = fem.fem_mesh_create(m, TP)
    try:
        fem.fem_mesh_tune(h, variant, 0)
        # (the kernels on stored hex matrices take the mesh's own coefficients only)
        coeffs = ((CM, CK),) if variant in (7, 9) else ((1.0, 0.0), (CM, CK))
        _check(torch_dev, fem.fem_ebe_apply, h, m, K, M, coeffs, 8, 2e-3 if variant == 9 else 2e-6)
    finally:
        fem.fem_mesh_destroy(h)
