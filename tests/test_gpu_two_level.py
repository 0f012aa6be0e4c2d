"""The two-level preconditioner: block-Jacobi plus a coarse correction on the
element-mean potential (through the C ABI).

* the coarse operator A0 = P^T J_PhiPhi(u) P, assembled on the GPU from seven
  coloured J v products, equals the same product formed from the oracle's
  assembled Jacobian, entry by entry, to 1e-12 of its largest entry, and has no
  entry outside the 7-point element stencil (the potential couples only
  face neighbours in the SIPG form of Sec. 3.3);
* FGMRES preconditioned by it reaches the tolerance on the true (oracle)
  residual and the direct-solve solution, in fewer iterations than with
  block-Jacobi alone, on one- to four-level hierarchies (grid-wide and
  one-block smoothing) and with FP32 vectors;
* with a singular coarse operator (no electrode fixes the potential) the
  coarsest level falls back to smoothing and FGMRES still converges;
* Newton with it reaches the oracle's Newton solution;
* argument errors are reported.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def _enp():
    import paper_2112_09271_gb300 as enp
    enp.build()
    return enp


def _cuda(x):
    import torch
    return torch.tensor(np.asarray(x), device="cuda")


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _a0_oracle(orc, P, u):
    """P^T J_PhiPhi P from the oracle's assembled Jacobian (dense, E x E)."""
    import scipy.sparse as sp
    J = orc.jacobian(u).tocsr()
    nphi = P.E * P.Np
    Pm = sp.csr_matrix((np.ones(nphi), (np.arange(nphi), np.repeat(np.arange(P.E), P.Np))),
                       shape=(nphi, P.E))
    return (Pm.T @ J[:nphi, :nphi] @ Pm).toarray()


def _a0_dense(P, st):
    """Dense E x E matrix from the stencil rows [E][7] (self, -x, +x, -y, +y, -z, +z)."""
    nx, ny, nz = P.n_el
    A = np.zeros((P.E, P.E))
    off = [0, -1, 1, -nx, nx, -nx * ny, nx * ny]
    for K in range(P.E):
        ix, iy, iz = K % nx, (K // nx) % ny, K // (nx * ny)
        ok = [True, ix > 0, ix < nx - 1, iy > 0, iy < ny - 1, iz > 0, iz < nz - 1]
        for d in range(7):
            if ok[d]:
                A[K, K + off[d]] += st[K, d]
            else:
                assert st[K, d] == 0.0
    return A


@pytest.mark.parametrize("cfg,p,batch", [("channel_n2", 2, 1), ("cube_n3_p3", None, 1),
                                         ("reactor_n1_p2", None, 2)])
def test_coarse_operator_matches_oracle(cfg, p, batch):
    enp = _enp()
    P = W.config(cfg, p=p) if p else W.config(cfg)
    phis = [[1.17 + 0.5 * i, 0.0, 0.0, 0.0] for i in range(batch)]
    us = [W.random_state(P, 2 + i) for i in range(batch)]
    op = enp.Operator(P, batch=batch)
    if batch > 1:
        op.set_phi_app(np.array(phis))
    op.set_preconditioner(1)
    op.block_jacobi_setup(_cuda(np.concatenate(us)), 0)
    a0 = op.coarse_operator().cpu().numpy().reshape(batch, P.E, 7)
    for i in range(batch):
        Pi = dataclasses.replace(P, bv_phi_app=phis[i]) if batch > 1 else P
        ref = _a0_oracle(oracle.Oracle(Pi), Pi, us[i])
        got = _a0_dense(P, a0[i])
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


def _solve(op, u, b, two_level, f32=False, restart=60, max_it=4000, rtol=1e-10):
    import torch
    op.set_preconditioner(1 if two_level else 0)
    ud = _cuda(u)
    op.block_jacobi_setup(ud, 0 if not f32 else 1)
    dt = torch.float32 if f32 else torch.float64
    x = torch.zeros(b.size, dtype=dt, device="cuda")
    st = op.fgmres_solve(ud.to(dt), _cuda(b).to(dt), x, restart=restart, max_it=max_it, rtol=rtol)
    return x.double().cpu().numpy(), st


# cube_n21_p1: 9261 cells on the finest coarse level, above the one-block
# V-cycle's 8192, so its smoothing runs grid-wide and the levels below in one block
@pytest.mark.parametrize("cfg,levels", [("cube_n5_p2", 1), ("cube_n9_p1", 2),
                                        ("cube_n18_p1", 3), ("cube_n21_p1", 4)])
def test_two_level_fgmres_converges_faster(cfg, levels):
    enp = _enp()
    P = W.config(cfg)
    nx = P.n_el[0]
    n_lev, m = 1, nx
    while m ** 3 > 128:  # coarsest grid: at most 128 cells, solved with its inverse
        m, n_lev = (m + 1) // 2, n_lev + 1
    assert n_lev == levels
    orc = oracle.Oracle(P)
    u = W.random_state(P, 2)
    b = W.random_vector(P, 6)
    op = enp.Operator(P)
    x1, st1 = _solve(op, u, b, False)
    x2, st2 = _solve(op, u, b, True)
    assert st1["converged"] == 1 and st2["converged"] == 1
    for x in (x1, x2):
        assert np.linalg.norm(orc.jvp(u, x) - b) <= 1.01e-10 * np.linalg.norm(b)
    assert _rel(x2, x1) < 1e-6
    assert st2["iterations"] < st1["iterations"], (st1["iterations"], st2["iterations"])
    if P.n_dof < 30000:
        assert _rel(x2, orc.linear_solve(u, b)) < 1e-6


def test_singular_coarse_operator_falls_back_to_smoothing():
    """Without electrodes no boundary condition fixes the potential: a uniform
    shift of Phi leaves every flux unchanged, so A0 has the constant vector in
    its kernel (checked) and J is singular. The coarsest level then falls back
    from its inverse to Gauss-Seidel smoothing, and FGMRES still solves a
    consistent system J x = b (b = J x_true) to the tolerance."""
    import torch
    enp = _enp()
    P = W.config("cube_n9_p1")
    P = dataclasses.replace(P, tags=[np.where(t >= W.ELECTRODE0, W.WALL, t).astype(np.uint8)
                                   for t in P.tags])
    orc = oracle.Oracle(P)
    u = W.random_state(P, 2)
    b = orc.jvp(u, W.random_vector(P, 6))
    op = enp.Operator(P)
    op.set_preconditioner(1)
    ud = _cuda(u)
    op.block_jacobi_setup(ud, 0)
    a0 = op.coarse_operator().cpu().numpy().reshape(P.E, 7)
    assert np.abs(a0.sum(axis=1)).max() <= 1e-12 * np.abs(a0).max()
    x = torch.zeros(P.n_dof, dtype=torch.float64, device="cuda")
    st = op.fgmres_solve(ud, _cuda(b), x, restart=60, max_it=4000, rtol=1e-10)
    assert st["converged"] == 1
    assert np.linalg.norm(orc.jvp(u, x.cpu().numpy()) - b) <= 1.01e-10 * np.linalg.norm(b)


def test_two_level_fgmres_f32():
    enp = _enp()
    P = W.config("cube_n9_p1")
    orc = oracle.Oracle(P)
    u = W.random_state(P, 2)
    b = W.random_vector(P, 6)
    op = enp.Operator(P)
    x, st = _solve(op, u, b, True, f32=True, rtol=1e-5)
    assert st["converged"] == 1
    assert np.linalg.norm(orc.jvp(u, x) - b) <= 1e-4 * np.linalg.norm(b)


@pytest.mark.parametrize("mixed", [False, True])
def test_two_level_newton_matches_oracle_newton(mixed):
    enp = _enp()
    P = W.config("cube_n3_p2")
    orc = oracle.Oracle(P)
    u0 = np.zeros((P.n_fields, P.E, P.Np))
    for k in range(1, P.n_fields):
        u0[k] = P.c_in[k - 1]
    u0 = u0.reshape(-1)
    ref, _ = orc.newton_solve(u0, rtol=1e-12, max_it=30)
    op = enp.Operator(P)
    op.set_preconditioner(1)
    ud = _cuda(u0)
    st = op.newton_solve(ud, max_it=30, rtol=1e-10, krylov_rtol=1e-3 if not mixed else 1e-2,
                         bj_storage=0 if not mixed else 1, mixed=mixed)
    assert st["converged"] == 1, st
    assert _rel(ud.cpu().numpy(), ref) < 1e-8


def test_two_level_argument_errors():
    enp = _enp()
    op = enp.Operator(W.config("cube_n2_p2"))
    with pytest.raises(enp.EnpError) as ei:
        op.set_preconditioner(2)
    assert ei.value.status == enp.ENP_ERR_INVALID_ARG
    with pytest.raises(enp.EnpError) as ei:
        op.coarse_operator()  # not set up
    assert ei.value.status == enp.ENP_ERR_INVALID_ARG
    op2 = enp.Operator(W.config("mms2d_n3"))
    with pytest.raises(enp.EnpError) as ei:
        op2.set_preconditioner(1)
    assert ei.value.status == enp.ENP_ERR_UNSUPPORTED


@pytest.mark.parametrize("two_level", [0, 1])
def test_lagged_preconditioner_newton(two_level):
    """A preconditioner rebuilt every third Newton iteration (pc_lag = 3) still
    gives the oracle's Newton solution; the setups counted are ceil(its / 3)
    when every inner solve converged."""
    enp = _enp()
    P = W.config("cube_n3_p2")
    orc = oracle.Oracle(P)
    u0 = np.zeros((P.n_fields, P.E, P.Np))
    for k in range(1, P.n_fields):
        u0[k] = P.c_in[k - 1]
    u0 = u0.reshape(-1)
    ref, _ = orc.newton_solve(u0, rtol=1e-12, max_it=30)
    op = enp.Operator(P)
    op.set_preconditioner(two_level)
    ud = _cuda(u0)
    st = op.newton_solve(ud, max_it=30, rtol=1e-10, krylov_rtol=1e-3, krylov_max_it=2000,
                         pc_lag=3)
    assert st["converged"] == 1, st
    assert st["setups"] == -(-st["iterations"] // 3)
    assert st["setup_seconds"] > 0 and st["krylov_seconds"] > 0
    assert _rel(ud.cpu().numpy(), ref) < 1e-8


def test_two_level_graph_equals_eager_batched():
    """The coarse correction is captured with the rest of a restart cycle: the
    graph-replayed batched FGMRES gives bit for bit the eager iterate."""
    import torch
    enp = _enp()
    P = W.config("reactor_n1_p2")
    B = 2
    phis = np.array([[1.0, 0, 0, 0], [3.0, 0, 0, 0]])
    u = _cuda(np.concatenate([W.random_state(P, 2), W.random_state(P, 3)]))
    b = _cuda(np.concatenate([W.random_vector(P, 6), 10 * W.random_vector(P, 7)]))
    op = enp.Operator(P, batch=B)
    op.set_phi_app(phis)
    op.set_preconditioner(1)
    op.block_jacobi_setup(u, 0)
    xs, its = [], []
    for graph in (False, True):
        x = torch.zeros(B * P.n_dof, dtype=torch.float64, device="cuda")
        st = op.fgmres_solve(u, b, x, restart=30, max_it=600, rtol=1e-10, graph=graph)
        assert st["converged"] == 1
        xs.append(x.cpu().numpy())
        its.append(st["iterations"])
    np.testing.assert_array_equal(xs[0], xs[1])


def _vcycle(A, b, smooth=2, omega=1.8):
    """One V-cycle in FP64 on the packed stencil A [nz, ny, nx, 7]."""
    def off(t):
        o = np.zeros_like(t)
        o[:, :, 1:] += A[:, :, 1:, 1] * t[:, :, :-1]
        o[:, :, :-1] += A[:, :, :-1, 2] * t[:, :, 1:]
        o[:, 1:] += A[:, 1:, :, 3] * t[:, :-1]
        o[:, :-1] += A[:, :-1, :, 4] * t[:, 1:]
        o[1:] += A[1:, :, :, 5] * t[:-1]
        o[:-1] += A[:-1, :, :, 6] * t[1:]
        return o

    n = b.size
    if n <= 128:
        M = np.empty((n, n))
        for i in range(n):
            e = np.zeros(n)
            e[i] = 1.0
            e = e.reshape(b.shape)
            M[:, i] = (A[..., 0] * e + off(e)).reshape(-1)
        return np.linalg.solve(M, b.reshape(-1)).reshape(b.shape)
    iz, iy, ix = np.indices(b.shape)
    par = (ix + iy + iz) % 2
    x = np.zeros_like(b)
    for c in (0, 1) * smooth:
        x = np.where(par == c, (b - off(x)) / A[..., 0], x)
    res = b - A[..., 0] * x - off(x)
    c = tuple((k + 1) // 2 for k in b.shape)
    Ac, bc = np.zeros(c + (7,)), np.zeros(c)
    np.add.at(bc, (iz // 2, iy // 2, ix // 2), res)
    inside = {1: ix % 2 == 1, 2: ix % 2 == 0, 3: iy % 2 == 1, 4: iy % 2 == 0, 5: iz % 2 == 1,
              6: iz % 2 == 0}
    at = (iz // 2, iy // 2, ix // 2)
    np.add.at(Ac[..., 0], at, A[..., 0])
    for d in range(1, 7):
        np.add.at(Ac[..., 0], at, np.where(inside[d], A[..., d], 0.0))
        np.add.at(Ac[..., d], at, np.where(inside[d], 0.0, A[..., d]))
    x = x + omega * _vcycle(Ac, bc, smooth, omega)[at]
    for c in (1, 0) * smooth:
        x = np.where(par == c, (b - off(x)) / A[..., 0], x)
    return x


@pytest.mark.parametrize("smooth", [1, 2])
@pytest.mark.parametrize("n", [(5, 5, 5), (12, 11, 10), (13, 13, 13), (33, 32, 32)])
def test_vcycle_of_every_level_size(n, smooth):
    """The coarse correction against a V-cycle in FP64 on the exported stencil: the
    coarsest level alone, levels in one block's shared memory (up to 2,048 cells),
    in the cluster (up to 32,768) and in grid-wide launches, odd sizes among them.
    FP32 arithmetic and an inverse stored in FP32: unit roundoff 6e-8 times a
    condition number of the coarsest matrix of at most some 1e3, so 2e-4."""
    import dataclasses
    enp = _enp()
    base = W.config("cube_n2_p2", p=1)
    coords = [np.linspace(0.0, 1.0, k + 1) for k in n]
    tags = W.box_tags(3, list(n), coords, W.WALL)
    tags[0][:], tags[1][:] = W.INLET, W.OUTLET
    tags[2][:], tags[3][:] = W.ELECTRODE0, W.ELECTRODE0 + 1
    P = dataclasses.replace(base, n_el=list(n), coords=coords, tags=tags)
    op = enp.Operator(P)
    u, r = _cuda(W.random_state(P, 1)), W.random_vector(P, 2)
    op.set_coarse_options(cycles=1, smooth=smooth, omega=1.8)
    op.set_preconditioner(1)
    op.block_jacobi_setup(u, enp.BJ_F64)
    with_ = op.block_jacobi_apply(_cuda(r)).cpu().numpy()
    A = op.coarse_operator().cpu().numpy().reshape(n[2], n[1], n[0], 7)
    op.set_preconditioner(0)
    op.block_jacobi_setup(u, enp.BJ_F64)
    plain = op.block_jacobi_apply(_cuda(r)).cpu().numpy()
    d = (with_ - plain).reshape(P.n_fields, P.E, P.Np)
    assert not d[1:].any()
    b = r.reshape(P.n_fields, P.E, P.Np)[0].sum(-1).reshape(n[2], n[1], n[0])
    ref = _vcycle(A, b, smooth).reshape(-1)
    assert np.linalg.norm(d[0, :, 0] - ref) <= 2e-4 * np.linalg.norm(ref)
    assert np.abs(d[0] - d[0, :, :1]).max() <= 1e-12 * np.abs(with_).max()


# one element's potential residuals whose sum needs 53 bits, and whose partial sums
# pass FP32's range: FP64 forms both exactly, in any order
@pytest.mark.parametrize("values,total", [
    ([1.0, 2.0 ** -26, 2.0 ** -52, -1.0, -2.0 ** -26], 2.0 ** -52),
    ([3e38, 3e38, -3e38, -3e38], 0.0)])
@pytest.mark.parametrize("cfg", ["cube_n5_p2", "cube_n5_p3"])   # one lane an element, four
def test_coarse_right_hand_side_is_summed_in_fp64(cfg, values, total):
    """FP32 vectors: P^T r is summed in FP64, so a residual in one element equals, in
    every other element (where the block part is zero), bit for bit the coarse
    correction of a residual that is that sum at one node."""
    enp = _enp()
    P = W.config(cfg)
    op = enp.Operator(P)
    op.set_preconditioner(1)
    op.set_sweep(0)
    op.block_jacobi_setup(_cuda(W.random_state(P, 2)), enp.BJ_F32)
    K = P.E // 2
    z = []
    for v in (values, [total]):
        r = np.zeros((P.n_fields, P.E, P.Np), np.float32)
        r[0, K, :4 * len(v):4] = v     # of one lane
        z.append(op.block_jacobi_apply_f32(_cuda(r.reshape(-1))).cpu().numpy().reshape(r.shape))
    others = np.arange(P.E) != K
    assert (np.abs(z[1][0, others]).max() > 0) == (total != 0)
    np.testing.assert_array_equal(z[0][:, others], z[1][:, others])


@pytest.mark.parametrize("batch", [9, 20, 40, 80])
@pytest.mark.parametrize("n", [(6, 6, 6), (13, 13, 13)])
def test_vcycle_of_many_points_equals_each_alone(n, batch):
    """The blocks that share a point's V-cycle are as many as run at once for the whole
    batch (one to eight), and do not change a bit of any point's correction."""
    import dataclasses
    enp = _enp()
    base = W.config("cube_n2_p2", p=1)
    coords = [np.linspace(0.0, 1.0, k + 1) for k in n]
    tags = W.box_tags(3, list(n), coords, W.WALL)
    tags[0][:], tags[1][:] = W.INLET, W.OUTLET
    tags[2][:] = W.ELECTRODE0
    P = dataclasses.replace(base, n_el=list(n), coords=coords, tags=tags)
    us = [W.random_state(P, 2 + i % 5) for i in range(batch)]
    rs = [W.random_vector(P, 3 + i % 7) for i in range(batch)]

    def corrections(u, r, b):
        op = enp.Operator(P, batch=b)
        op.set_preconditioner(1)
        op.block_jacobi_setup(_cuda(u), enp.BJ_F32)
        return op.block_jacobi_apply_f32(_cuda(r).float()).cpu().numpy().reshape(b, -1)

    z = corrections(np.concatenate(us), np.concatenate(rs), batch)
    for i in (0, 1, batch // 2, batch - 1):
        np.testing.assert_array_equal(z[i], corrections(us[i], rs[i], 1)[0])


def test_two_level_fgmres_with_grid_wide_smoothing():
    """35,937 cells: the finest level's smoothing runs in launches over the whole grid,
    the levels below in one. FGMRES reaches the tolerance on the oracle's residual, in a
    number of iterations that block-Jacobi alone does not do with."""
    import torch
    enp = _enp()
    P = W.config("cube_n33_p1")
    assert P.E > 32768
    orc = oracle.Oracle(P)
    u, b = W.random_state(P, 2), W.random_vector(P, 6)
    op = enp.Operator(P)
    x, st = _solve(op, u, b, True)
    assert st["converged"] == 1
    assert np.linalg.norm(orc.jvp(u, x) - b) <= 1.01e-10 * np.linalg.norm(b)
    op.set_preconditioner(0)
    op.block_jacobi_setup(_cuda(u), enp.BJ_F64)
    y = torch.zeros(b.size, dtype=torch.float64, device="cuda")
    st = op.fgmres_solve(_cuda(u), _cuda(b), y, restart=60, max_it=st["iterations"], rtol=1e-10,
                         raise_on_fail=False)
    assert st["status"] == enp.ENP_ERR_NOT_CONVERGED
