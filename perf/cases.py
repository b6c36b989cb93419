"""Timed cases of the framework: what its users have it do, through its public entry points.

A case is a dict of plain values.  `kind` names the entry point:

  ebe    fem_ebe_apply: the matrix-free product q = A p of linear tets (optionally with the fused p^T q)
  ebe10  fem_ebe10_apply: the same product on 10-node tets
  split  fem_mesh_split_product in double-float arithmetic: M p and K p, the certification product
  pcg    pcg_solve: one block-Jacobi PCG solve from a zero guess
  step   fem_step: time steps of a batch of cases (predict, right-hand side, certified solve, update)
  mlp    fem_mlp_loss_grad: forward and backward pass of the learned proposal's network

Meshes are the seeded recipes of `workload`: three log-normal layers ("layered"), five layers with a basin
("basin"), two layers on the unit box ("unit"), and "tets": the layered recipe with moved interior nodes and
the elements in an order with locality but no six tets of a hexahedron in a row, as an unstructured mesher
hands them over.  nx, ny, nz are hexahedra (six tets each), r the number of cases solved together.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2409_20380_gb300 import fem
from paper_2409_20380_gb300 import workload as wl

DEV = "cuda"


def listed():
    return [
        # the smallest call: the product on the unit box of 3072 tets, one case, where latency and launches count
        dict(name="ebe_unit", kind="ebe", mesh="unit", nx=8, ny=8, nz=8, r=1, f64=False, ptq=False),
        # the inner solve's product on the medium workload: 16 cases, with the fused p^T A p
        dict(name="ebe_medium", kind="ebe", mesh="layered", nx=64, ny=64, nz=32, r=16, f64=False, ptq=True),
        # the same on the large recipe (6.3 M tets), 8 cases
        dict(name="ebe_large", kind="ebe", mesh="basin", nx=128, ny=128, nz=64, r=8, f64=False, ptq=True),
        # a ragged box of the uneven-mesh workload's range, two cases
        dict(name="ebe_uneven", kind="ebe", mesh="layered", nx=57, ny=39, nz=31, r=2, f64=False, ptq=False),
        # a mesh without hexahedral patches: any tetrahedral mesh a user brings
        dict(name="ebe_tets", kind="ebe", mesh="tets", nx=53, ny=45, nz=27, r=8, f64=False, ptq=False),
        # the quadratic element on the medium grid, 16 cases
        dict(name="ebe10_medium", kind="ebe10", mesh="layered", nx=64, ny=64, nz=32, r=16, f64=False),
        # the product every step is certified with, medium workload
        dict(name="split_medium", kind="split", mesh="layered", nx=64, ny=64, nz=32, r=16),
        # a tight solve (FP32 inside, FP64 outside) on a ragged box, from nothing
        dict(name="pcg_uneven", kind="pcg", mesh="layered", nx=49, ny=61, nz=37, r=4, f64=False, tol=1e-12),
        # one training pass of the learned proposal at its training batch
        dict(name="mlp_train", kind="mlp", batch=4096),
        # the tiny workload: one case in FP64, where a step is launches and host work
        dict(name="step_unit", kind="step", mesh="unit", nx=8, ny=8, nz=8, r=1, f64=True, s=8, steps=10, spinup=40),
        # the medium workload: 16 cases, 32 stored pairs, FP32 inside, certified in FP64
        dict(name="step_medium", kind="step", mesh="layered", nx=64, ny=64, nz=32, r=16, f64=False, s=32, steps=4,
             spinup=60),
        # the large recipe: 8 cases, 16 stored pairs, the inner products on the tensor cores as the benchmark has it
        dict(name="step_large", kind="step", mesh="basin", nx=128, ny=128, nz=64, r=8, f64=False, s=16, steps=2,
             spinup=60),
    ]


def _dims(rng, lo, hi):
    """A box of about 2 n^2 x n/2-like proportions with lo..hi hexahedra (log-uniform), odd and ragged."""
    H = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nz = max(4, round((H / 4.0) ** (1.0 / 3.0) * rng.uniform(0.8, 1.25)))
    nx = max(4, round(math.sqrt(H / nz) * rng.uniform(0.8, 1.25)))
    ny = max(4, int(H / (nz * nx)))
    return nx, ny, nz


def draw(rng):
    kind = rng.choice(["ebe", "ebe", "ebe", "ebe", "ebe10", "split", "pcg", "mlp", "step", "step"])
    if kind == "mlp":
        return dict(kind="mlp", batch=round(math.exp(rng.uniform(math.log(256), math.log(16384)))))
    r = rng.choice([1, 2, 4, 8, 16, 32] if kind == "ebe" else [1, 2, 4, 8, 16])
    top = {"ebe": 8388608 // r, "ebe10": 2097152 // r, "split": 2097152 // r, "pcg": 524288 // r, "step": 2097152 // r}
    nx, ny, nz = _dims(rng, 512, min(top[kind], 1048576 if kind == "ebe" else 131072))
    case = dict(kind=kind, mesh="layered", nx=nx, ny=ny, nz=nz, r=r)
    if kind == "ebe":
        case["mesh"] = rng.choice(["layered", "layered", "basin", "tets"])
        case["f64"] = rng.random() < 0.2
        case["ptq"] = rng.random() < 0.5 and 6 * nx * ny * nz * r > 4000000
    elif kind == "ebe10":
        case["f64"] = False
    elif kind == "pcg":
        case["f64"] = rng.random() < 0.3
        case["tol"] = 1e-12
    elif kind == "step":
        case.update(mesh=rng.choice(["layered", "basin"]), f64=False, s=rng.choice([8, 16, 32]), steps=4, spinup=60)
    return case


# --- inputs ------------------------------------------------------------------------------------------------


def _time_params(kind):
    return wl.TimeParams() if kind == "unit" else wl.config2_time_params()


@functools.lru_cache(maxsize=2)
def _host_mesh(kind, nx, ny, nz):
    if kind == "unit":
        return wl.config1_mesh()
    if kind == "basin":
        return wl.config4_mesh(nx, ny, nz)
    m = wl.config2_mesh(nx, ny, nz)
    if kind == "tets":
        rng = np.random.default_rng([20380, nx, ny, nz])
        inner = wl.interior_nodes(m)
        m.xyz[inner] += 0.15 * m.h * rng.uniform(-1.0, 1.0, (inner.size, 3))
        order = np.argsort(np.arange(m.n_elems) + rng.uniform(0.0, 96.0, m.n_elems), kind="stable")
        m.conn = np.ascontiguousarray(m.conn[order])
        m.mat_id = np.ascontiguousarray(m.mat_id[order])
    return m


@functools.lru_cache(maxsize=1)
def _host_mesh10(kind, nx, ny, nz):
    return wl.tet10_mesh_ordered(_host_mesh(kind, nx, ny, nz))[0]


@functools.lru_cache(maxsize=2)
def _host_regions(kind, nx, ny, nz):
    return wl.region_map(_host_mesh(kind, nx, ny, nz), 1024)


def _mesh_of(case):
    key = (case["mesh"], case["nx"], case["ny"], case["nz"])
    return _host_mesh10(*key) if case["kind"] == "ebe10" else _host_mesh(*key)


def _system(tp):
    """Coefficients of A = cM M + cK K."""
    return 4.0 / tp.dt ** 2 + 2.0 * tp.a0 / tp.dt, 1.0 + 2.0 * tp.a1 / tp.dt


def _vectors(mesh, r, seed, dtype):
    """Random nodal vectors [N][3][r], zero on Dirichlet DOFs."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    free = torch.from_numpy(mesh.fixed_dof == 0).to(DEV).to(dtype)
    v = torch.randn((3 * mesh.n_nodes, r), generator=g, device=DEV, dtype=dtype)
    return (v * free[:, None]).reshape(-1)


def _sources(case, mesh, seed):
    rngs = [np.random.default_rng([seed, c]) for c in range(case["r"])]
    return [wl.random_source(mesh, g, f0=5.0 if case["mesh"] == "unit" else None) for g in rngs]


def _mlp_inputs(case, seed):
    """Features, targets and weights of the sizes the time steps collect: 36 used inputs of order one, coefficient
    corrections well below the coefficients."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    B = case["batch"]
    x = torch.randn((B, 64), generator=g, device=DEV)
    x[:, 36:] = 0.0
    t = 0.3 * torch.randn((B, 32), generator=g, device=DEV)
    return x, t, wl.mlp_init_weights(seed).astype(np.float32)


class _State:
    """What a user's program holds: handles and device buffers, given back together."""

    def __init__(self, case):
        self.case = case
        self.given_back = []

    def keep(self, handle, destroy):
        self.given_back.append((destroy, handle))
        return handle

    def __del__(self):
        if self.given_back:
            torch.cuda.synchronize()
        while self.given_back:
            destroy, handle = self.given_back.pop()
            destroy(handle)


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "mlp":
        s.x, s.t, theta = _mlp_inputs(case, seed)
        s.net = s.keep(fem.fem_mlp_create(theta), fem.fem_mlp_destroy)
        s.grad = torch.empty(fem.FEM_MLP_N_PARAMS, device=DEV)
        return s
    mesh, tp = _mesh_of(case), _time_params(case["mesh"])
    s.cM, s.cK = _system(tp)
    r = case["r"]
    if kind == "ebe10":
        s.mesh = s.keep(fem.fem_mesh10_create(mesh), fem.fem_mesh10_destroy)
    else:
        s.mesh = s.keep(fem.fem_mesh_create(mesh, tp), fem.fem_mesh_destroy)
    if kind == "step":
        s.n = mesh.n_nodes
        fem.fem_mesh_set_regions(s.mesh, _host_regions(case["mesh"], case["nx"], case["ny"], case["nz"]))
        tc = case["mesh"] == "basin" and 5 <= r <= 16
        s.batch = s.keep(fem.fem_batch_create(fem.fem_opts_default(
            precision=fem.FEM_FP64 if case["f64"] else fem.FEM_FP32_INNER, predictor=fem.FEM_PRED_DD, s_max=case["s"],
            inner_product=fem.FEM_INNER_TC if tc else fem.FEM_INNER_FP32)), fem.fem_batch_destroy)
        for src in _sources(case, mesh, seed):
            fem.fem_case_add(s.batch, s.mesh, src)
        fem.fem_step(s.batch, case["spinup"], r)
        s.fields = [torch.empty(r * s.n * 3, dtype=torch.float64, device=DEV) for _ in range(3)]
        return s
    dtype = torch.float64 if kind in ("split", "pcg") or case["f64"] else torch.float32
    s.p = _vectors(mesh, r, seed, dtype)
    s.q = torch.empty_like(s.p)
    if kind == "split":
        s.q2 = torch.empty_like(s.p)
    elif kind == "pcg":
        s.opts = fem.fem_opts_default(precision=fem.FEM_FP64 if case["f64"] else fem.FEM_FP32_INNER, tol=case["tol"])
    elif kind == "ebe":
        s.ptq = torch.empty(r, dtype=torch.float64, device=DEV) if case["ptq"] else None
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "ebe":
        fem.fem_ebe_apply(s.mesh, s.p, s.q, s.case["r"], s.cM, s.cK, s.ptq)
        return [s.q] if s.ptq is None else [s.q, s.ptq]
    if kind == "ebe10":
        fem.fem_ebe10_apply(s.mesh, s.p, s.q, s.case["r"], s.cM, s.cK)
        return [s.q]
    if kind == "split":
        fem.fem_mesh_split_product(s.mesh, 3, s.p, s.q, s.q2, s.case["r"])
        return [s.q, s.q2]
    if kind == "pcg":
        s.q.zero_()
        fem.pcg_solve(s.mesh, s.p, s.q, s.case["r"], s.opts)
        return [s.q]
    if kind == "mlp":
        return [s.grad, fem.fem_mlp_loss_grad(s.net, s.x, s.t, s.grad)]
    fem.fem_step(s.batch, s.case["steps"], s.case["r"])
    for what, field in zip((fem.FEM_FIELD_U, fem.FEM_FIELD_V, fem.FEM_FIELD_A), s.fields):
        fem.fem_batch_get_field(s.batch, what, field)
    return s.fields


def work(case):
    """Each tet's node ids (4 bytes each) and material id and the node coordinates read once, the nodal vectors
    read and written once; 190 operations a linear tet and case, 1570 a quadratic one (the gradient, stress and
    force sums and the consistent mass).  A CG iteration also reads and writes its three vectors once."""
    kind = case["kind"]
    if kind == "mlp":
        B, W = case["batch"], 64 * 256 + 256 * 256 + 256 * 32
        return {"bytes": B * (64 + 32) * 4 + 2 * 4 * fem.FEM_MLP_N_PARAMS, "flops": 6 * B * W}
    nx, ny, nz, r = case["nx"], case["ny"], case["nz"], case["r"]
    E, N = 6 * nx * ny * nz, (nx + 1) * (ny + 1) * (nz + 1)
    if kind == "ebe10":
        N10 = (2 * nx + 1) * (2 * ny + 1) * (2 * nz + 1)
        return {"bytes": E * 44 + N10 * (24 + 2 * 3 * r * 4), "flops": 1570 * E * r}
    word = 8 if kind == "split" or case["f64"] else 4
    V = 3 * N * r
    mesh = E * 20 + N * 24
    if kind == "ebe":
        return {"bytes": mesh + 2 * V * word, "flops": 190 * E * r}
    if kind == "split":
        return {"bytes": mesh + 3 * V * 8, "flops": 200 * E * r}
    iters = 40 if kind == "pcg" else 6                       # typical counts of these solves
    solve = {"bytes": 2 * V * 8 + iters * (mesh + 8 * V * word), "flops": iters * r * (190 * E + 40 * N)}
    if kind == "pcg":
        return solve
    pairs = 2 * case["s"] * V * 8 + 12 * V * 8               # the stored pairs and the state, once a step
    return {"bytes": case["steps"] * (solve["bytes"] + pairs), "flops": case["steps"] * (solve["flops"] + 8 * case["s"] * V)}


# --- the same results in 64 bits, from the textbook forms ------------------------------------------------------


def _tet_geometry(mesh, conn):
    """Barycentric gradients [E][4][3], volume, lambda, mu, rho of every element, on the GPU."""
    xyz = torch.from_numpy(mesh.xyz).to(DEV)
    x = xyz[conn[:, :4]]
    J = x[:, 1:] - x[:, :1]                                  # rows: edges from corner 0
    g123 = torch.linalg.inv(J).transpose(1, 2)               # d(xi_k)/dx as rows
    g = torch.cat([-g123.sum(1, keepdim=True), g123], 1)
    V = torch.linalg.det(J) / 6.0
    lmr = torch.from_numpy(mesh.lam_mu_rho).to(DEV)[torch.from_numpy(mesh.mat_id).to(DEV).long()]
    return g, V, lmr[:, 0], lmr[:, 1], lmr[:, 2]


def _mass10():
    """10 x 10 consistent mass of a straight-sided quadratic tet, times 420 / (rho V)."""
    edges = wl.TET10_EDGES
    m = np.ones((10, 10))
    for i in range(4):
        m[i, i] = 6.0
        for k, e in enumerate(edges):
            m[i, 4 + k] = m[4 + k, i] = -4.0 if i in e else -6.0
    for k, e in enumerate(edges):
        for l, f in enumerate(edges):
            m[4 + k, 4 + l] = 32.0 if k == l else 8.0 if not set(e) & set(f) else 16.0
    return torch.from_numpy(m).to(DEV) / 420.0


def _apply(mesh, p, r):
    """M p and K p, element by element: p [3N][r] -> two tensors of that shape (zero on Dirichlet DOFs)."""
    conn = torch.from_numpy(mesh.conn).to(DEV).long()
    n_loc = conn.shape[1]
    p = p.reshape(-1, 3, r)
    qM, qK = torch.zeros_like(p), torch.zeros_like(p)
    g, V, lam, mu, rho = _tet_geometry(mesh, conn)
    if n_loc == 4:
        m = (torch.ones((4, 4), dtype=torch.float64, device=DEV) + torch.eye(4, dtype=torch.float64, device=DEV)) / 20.0
        rules = [(1.0, None)]
    else:
        m = _mass10()
        a, b = (5.0 + 3.0 * math.sqrt(5.0)) / 20.0, (5.0 - math.sqrt(5.0)) / 20.0
        rules = [(0.25, [a if k == q else b for k in range(4)]) for q in range(4)]
    step = max(4096, (1 << 24) // (n_loc * 3 * r))
    for e0 in range(0, conn.shape[0], step):
        s = slice(e0, e0 + step)
        c, ge, Ve = conn[s], g[s], V[s]
        u = p[c]                                             # [e][a][i][case]
        fM = torch.einsum("ab,ebic->eaic", m, u) * (rho[s] * Ve)[:, None, None, None]
        fK = torch.zeros_like(u)
        for wq, L in rules:
            if L is None:
                dN = ge
            else:
                dN = torch.stack([(4.0 * L[a] - 1.0) * ge[:, a] for a in range(4)]
                                 + [4.0 * (L[a] * ge[:, b] + L[b] * ge[:, a]) for a, b in wl.TET10_EDGES], 1)
            G = torch.einsum("eaj,eaic->eijc", dN, u)
            S = mu[s][:, None, None, None] * (G + G.transpose(1, 2))
            tr = lam[s][:, None] * (G[:, 0, 0] + G[:, 1, 1] + G[:, 2, 2])
            for i in range(3):
                S[:, i, i] += tr
            fK += torch.einsum("eaj,eijc->eaic", dN, S) * (wq * Ve)[:, None, None, None]
        idx = c.reshape(-1)
        qM.index_add_(0, idx, fM.reshape(-1, 3, r))
        qK.index_add_(0, idx, fK.reshape(-1, 3, r))
    free = torch.from_numpy(mesh.fixed_dof == 0).to(DEV).reshape(-1, 3, 1)
    return (qM * free).reshape(-1, r), (qK * free).reshape(-1, r)


def _assembled(mesh):
    """M and K as sparse matrices [3N][3N] (Dirichlet rows and columns zero), linear tets."""
    conn = torch.from_numpy(mesh.conn).to(DEV).long()
    g, V, lam, mu, rho = _tet_geometry(mesh, conn)
    eye3 = torch.eye(3, dtype=torch.float64, device=DEV)
    gg = torch.einsum("eai,ebj->eaibj", g, g)
    Ke = lam[:, None, None, None, None] * gg + mu[:, None, None, None, None] * gg.transpose(2, 4)
    Ke = Ke + (mu[:, None, None] * torch.einsum("eai,ebi->eab", g, g))[:, :, None, :, None] * eye3[None, None, :, None, :]
    Ke = Ke * V[:, None, None, None, None]
    m4 = (torch.ones((4, 4), dtype=torch.float64, device=DEV) + torch.eye(4, dtype=torch.float64, device=DEV)) / 20.0
    Me = (rho * V)[:, None, None, None, None] * m4[None, :, None, :, None] * eye3[None, None, :, None, :]
    dof = (3 * conn[:, :, None] + torch.arange(3, device=DEV)).reshape(-1, 12)
    free = torch.from_numpy(mesh.fixed_dof == 0).to(DEV)
    keep = (free[dof][:, :, None] & free[dof][:, None, :]).reshape(-1)
    rows = dof[:, :, None].expand(-1, 12, 12).reshape(-1)[keep]
    cols = dof[:, None, :].expand(-1, 12, 12).reshape(-1)[keep]
    n = 3 * mesh.n_nodes
    out = []
    for B in (Me, Ke):
        out.append(torch.sparse_coo_tensor(torch.stack([rows, cols]), B.reshape(-1)[keep], (n, n)).coalesce().to_sparse_csr())
    return out


def _diagonal(mesh, cM, cK):
    """Diagonal of cM M + cK K (one on Dirichlet DOFs)."""
    conn = torch.from_numpy(mesh.conn).to(DEV).long()
    g, V, lam, mu, rho = _tet_geometry(mesh, conn)
    d = V[:, None, None] * ((lam + mu)[:, None, None] * g * g + mu[:, None, None] * (g * g).sum(2, keepdim=True))
    d = cK * d + (cM * rho * V / 10.0)[:, None, None]
    out = torch.zeros((mesh.n_nodes, 3), dtype=torch.float64, device=DEV).index_add_(0, conn.reshape(-1), d.reshape(-1, 3))
    free = torch.from_numpy(mesh.fixed_dof == 0).to(DEV)
    return torch.where(free, out.reshape(-1), torch.ones_like(out.reshape(-1)))


def _solve(A, dinv, b, x, tol):
    """Jacobi-preconditioned conjugate gradients of several right-hand sides in 64 bits."""
    bn = b.norm(dim=0).clamp_min(1e-300)
    res = b - A(x)
    z = dinv * res
    p, rz = z.clone(), (res * z).sum(0)
    for it in range(2000):
        if it % 4 == 0 and bool((res.norm(dim=0) / bn < tol).all()):
            break
        q = A(p)
        alpha = rz / (p * q).sum(0).clamp_min(1e-300)
        x = x + alpha * p
        res = res - alpha * q
        z = dinv * res
        new = (res * z).sum(0)
        p = z + (new / rz.clamp_min(1e-300)) * p
        rz = new
    return x


def _exact_steps(case, seed):
    mesh, tp, r = _mesh_of(case), _time_params(case["mesh"]), case["r"]
    cM, cK = _system(tp)
    M, K = _assembled(mesh)
    dinv = 1.0 / _diagonal(mesh, cM, cK)[:, None]
    free = torch.from_numpy(mesh.fixed_dof == 0).to(DEV).double()[:, None]

    def A(v):
        return cM * (M @ v) + cK * (K @ v)

    srcs = _sources(case, mesh, seed)
    u, v, a, du = (torch.zeros((3 * mesh.n_nodes, r), dtype=torch.float64, device=DEV) for _ in range(4))
    for it in range(1, case["spinup"] + case["steps"] + 1):
        f = torch.zeros_like(u)
        for c, s in enumerate(srcs):
            w = (math.pi * s.f0 * (it * tp.dt - s.t0)) ** 2
            f[3 * s.node:3 * s.node + 3, c] = torch.from_numpy(s.amp * (1.0 - 2.0 * w) * math.exp(-w) * s.direction).to(DEV)
        b = f * free - K @ u + tp.a0 * (M @ v) + tp.a1 * (K @ v) + M @ (a + 4.0 / tp.dt * v)
        du = _solve(A, dinv, b, du, 1e-13)
        u, v, a = u + du, 2.0 / tp.dt * du - v, 4.0 / tp.dt ** 2 * du - 4.0 / tp.dt * v - a
    return [w.T.reshape(-1) for w in (u, v, a)]


def _exact_mlp(case, seed):
    x, t, theta = _mlp_inputs(case, seed)
    x, t = x.double(), t.double()
    th = torch.from_numpy(theta).to(DEV).double().requires_grad_(True)
    sizes, o, a = (64, 256, 256, 32), 0, x
    for i in range(3):
        n_in, n_out = sizes[i], sizes[i + 1]
        W, b = th[o:o + n_in * n_out].reshape(n_out, n_in), th[o + n_in * n_out:o + n_in * n_out + n_out]
        o += n_in * n_out + n_out
        a = a @ W.T + b
        if i < 2:
            a = torch.nn.functional.gelu(a)
    loss = ((a - t) ** 2).mean()
    loss.backward()
    return [th.grad, float(loss.detach())]


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _exact_mlp(case, seed)
    if kind == "step":
        # the assembled matrices and 60 solves of more than this take over 20 seconds
        if 6 * case["nx"] * case["ny"] * case["nz"] * case["r"] > 16000000:
            return None
        return _exact_steps(case, seed)
    mesh, r = _mesh_of(case), case["r"]
    cM, cK = _system(_time_params(case["mesh"]))
    if kind == "pcg":
        M, K = _assembled(mesh)
        b = _vectors(mesh, r, seed, torch.float64).reshape(-1, r)
        dinv = 1.0 / _diagonal(mesh, cM, cK)[:, None]
        return [_solve(lambda v: cM * (M @ v) + cK * (K @ v), dinv, b, torch.zeros_like(b), 1e-14).reshape(-1)]
    dtype = torch.float64 if kind == "split" or case["f64"] else torch.float32
    p = _vectors(mesh, r, seed, dtype).double().reshape(-1, r)
    qM, qK = _apply(mesh, p, r)
    if kind == "split":
        return [qM.reshape(-1), qK.reshape(-1)]
    q = cM * qM + cK * qK
    return [q.reshape(-1), (p * q).sum(0)] if case.get("ptq") else [q.reshape(-1)]
