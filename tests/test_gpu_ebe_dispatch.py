"""The element products at the sizes where fem_ebe_apply's automatic choice changes: small meshes (the element
kernel with small blocks), the first tiled sizes, meshes without hex patches with pairs of cases, FP32 and FP64,
against the oracle's assembled matrix.  Bounds: a row's sum of ~60 FP32 contributions, each rounded a few times
(2^-24), relative to the largest entry: 2e-6; FP64 1e-13, the bounds of the other product tests."""
import numpy as np
import pytest

import oracle
from paper_2409_20380_gb300 import build, fem
from paper_2409_20380_gb300 import workload as wl
from helpers import from_cases, random_free_vectors, small_mesh, to_cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_dev():
    import torch
    build.build()
    fem.lib()
    return torch


def _check(torch, m, r, dtype, offset, tune=None):
    tp = wl.TimeParams()
    sysm, A = oracle.build_system(m, tp)
    cM, cK = 4.0 / tp.dt ** 2 + 2.0 * tp.a0 / tp.dt, 1.0 + 2.0 * tp.a1 / tp.dt
    vs = random_free_vectors(m, r, seed=r)
    h = fem.fem_mesh_create(m, tp)
    try:
        if tune:
            fem.fem_mesh_tune(h, *tune)
        n = 3 * m.n_nodes * r
        # offset 1: vectors that are not 8-byte (FP32) or 16-byte aligned
        p = torch.zeros(n + offset, dtype=dtype, device="cuda")[offset:]
        p.copy_(torch.tensor(from_cases(vs, m.n_nodes, r)))
        q = torch.full((n + offset,), float("nan"), dtype=dtype, device="cuda")[offset:]
        ptq = torch.empty(r, dtype=torch.float64, device="cuda")
        tol = 1e-13 if dtype == torch.float64 else 2e-6
        for red in (None, ptq):
            q.fill_(float("nan"))
            fem.fem_ebe_apply(h, p, q, r, cM, cK, red)
            for c, got in enumerate(to_cases(q.cpu().numpy().astype(np.float64), m.n_nodes, r)):
                x = to_cases(p.cpu().numpy().astype(np.float64), m.n_nodes, r)[c]
                ref = np.zeros(3 * m.n_nodes)
                ref[sysm.free] = A @ x[sysm.free]
                assert np.abs(got - ref).max() <= tol * np.abs(ref).max(), (r, c)
                assert np.all(got[m.fixed_dof == 1] == 0.0)
                if red is not None:
                    assert abs(float(ptq[c]) - x @ ref) <= tol * abs(x @ ref)
    finally:
        fem.fem_mesh_destroy(h)


# 16 x 16 x 16 hexes with 2 cases is the last FP32 size of the element kernel, 17 x 16 x 16 the first tiled one
@pytest.mark.parametrize("dims,r", [((1, 1, 1), 1), ((3, 2, 5), 32), ((8, 8, 8), 4), ((16, 16, 16), 2),
                                    ((17, 16, 16), 2), ((21, 20, 20), 1)])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("offset", [0, 1])
def test_automatic_choice(torch_dev, dims, r, dtype, offset):
    _check(torch_dev, small_mesh(*dims), r, getattr(torch_dev, dtype), offset)


@pytest.mark.parametrize("r", [1, 2, 4, 16])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("offset", [0, 1])
def test_no_hex_patches(torch_dev, r, dtype, offset):
    m = small_mesh(9, 7, 5, perturb=0.1)
    order = np.random.default_rng(3).permutation(m.n_elems)
    m.conn, m.mat_id = np.ascontiguousarray(m.conn[order]), np.ascontiguousarray(m.mat_id[order])
    _check(torch_dev, m, r, getattr(torch_dev, dtype), offset)


# Tile sizes that were asked for, at the edge of a block's shared memory: 490 nodes in a 256-hex tile (hexes in random
# order) fit the staged form but not the packed one with its own words; 64 hexes of 8 cases fit both.
@pytest.mark.parametrize("variant", [3, 5, 6])
@pytest.mark.parametrize("hpt", [64, 128, 256, 512])
@pytest.mark.parametrize("r", [4, 8, 16, 32])
def test_requested_tile_sizes(torch_dev, variant, hpt, r):
    m = small_mesh(6, 6, 9)
    order = np.random.default_rng(7).permutation(m.n_elems // 6)
    m.conn = np.ascontiguousarray(m.conn.reshape(-1, 6, 4)[order].reshape(-1, 4))
    m.mat_id = np.ascontiguousarray(m.mat_id.reshape(-1, 6)[order].reshape(-1))
    _check(torch_dev, m, r, torch_dev.float32, 0, (variant, hpt))
