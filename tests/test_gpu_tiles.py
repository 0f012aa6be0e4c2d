"""The hexahedral kernels at the edges of their thread groups.

A group of threads takes one to three elements (a warp one to three faces),
blocks hold several groups, and the last ones are partly empty: meshes of one
element, and of element and face counts that fill no group or block evenly, for
every degree and field count, against the FP64 oracle. Tolerances as in
test_gpu_operator.py: 1e-12 per field for the FP64-accurate operator (both
arithmetics), and for FP32 rounding 2e-5 per field.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def _problem(p, fields, n):
    base = W.config("cube_n2_p2" if fields == 2 else "channel_n1", p=p)
    L = [c[-1] for c in base.coords]
    # graded: the two sides of a face differ in size
    coords = [l * (np.linspace(0, 1, k + 1) ** 1.2) for l, k in zip(L, n)]
    tags = W.box_tags(3, list(n), coords, W.WALL)
    tags[0][:], tags[1][:] = W.INLET, W.OUTLET
    tags[2][:], tags[3][:] = W.ELECTRODE0, W.ELECTRODE0 + 1
    return dataclasses.replace(base, n_el=list(n), coords=coords, tags=tags)


def _rel(a, b, nf):
    a, b = np.asarray(a).reshape(nf, -1), np.asarray(b).reshape(nf, -1)
    return max(float(np.linalg.norm(x - y) / np.linalg.norm(y)) for x, y in zip(a, b))


@pytest.mark.parametrize("n", [(1, 1, 1), (5, 3, 1), (2, 1, 4)])
@pytest.mark.parametrize("fields", [2, 3])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_ragged_groups(p, fields, n):
    import torch
    import paper_2112_09271_gb300 as enp
    enp.build()
    P = _problem(p, fields, n)
    src = W.random_sources(P, 5)
    orc = oracle.Oracle(P, src=src)
    op = enp.Operator(P)
    op.set_sources(torch.tensor(src, device="cuda"), None)
    u, v, w = W.random_state(P, 1), W.random_vector(P, 2), W.random_vector(P, 3)
    ud, vd, wd = (torch.tensor(x, device="cuda") for x in (u, v, w))
    ref = (orc.residual(u), orc.jvp(u, v), orc.vjp_entries(u, w, np.arange(P.n_dof)))
    for arith in (enp.ARITH_F64, enp.ARITH_DF32):
        op.set_arithmetic(arith)
        got = (op.residual(ud), op.jvp(ud, vd), op.vjp(ud, wd))
        for g, r in zip(got, ref):
            assert _rel(g.cpu().numpy(), r, fields) < 1e-12
    jv = op.jvp_f32(ud.float(), vd.float()).cpu().numpy()
    u32, v32 = (x.float().double().cpu().numpy() for x in (ud, vd))
    assert _rel(jv, orc.jvp(u32, v32), fields) < 2e-5


@pytest.mark.parametrize("n", [(1, 1), (5, 3), (2, 7)])
@pytest.mark.parametrize("fields", [2, 3])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_quads(p, fields, n):
    """Quadrilaterals: one element, odd meshes, every degree and field count, with
    every boundary kind (Dirichlet on one side), FP64 and FP32."""
    import torch
    import paper_2112_09271_gb300 as enp
    enp.build()
    base = W.config("cube_n2_p2" if fields == 2 else "channel_n1", p=p)
    coords = [c[-1] * np.linspace(0, 1, k + 1) ** 1.2 for c, k in zip(base.coords, n)]
    tags = W.box_tags(2, list(n), coords, W.WALL)
    tags[0][:], tags[1][:] = W.INLET, W.OUTLET
    tags[2][:], tags[3][:] = W.ELECTRODE0, W.DIRICHLET
    P = dataclasses.replace(base, dim=2, n_el=list(n) + [1], coords=coords, tags=tags)
    src, dirv = W.random_sources(P, 5), W.random_dirichlet(P, 6)
    orc = oracle.Oracle(P, src=src, dirichlet=dirv)
    op = enp.Operator(P)
    op.set_sources(torch.tensor(src, device="cuda"), torch.tensor(dirv, device="cuda"))
    u, v, w = W.random_state(P, 1), W.random_vector(P, 2), W.random_vector(P, 3)
    ud, vd, wd = (torch.tensor(x, device="cuda") for x in (u, v, w))
    for g, r in ((op.residual(ud), orc.residual(u)), (op.jvp(ud, vd), orc.jvp(u, v)),
                 (op.vjp(ud, wd), orc.vjp_entries(u, w, np.arange(P.n_dof)))):
        assert _rel(g.cpu().numpy(), r, fields) < 1e-12
    jv = op.jvp_f32(ud.float(), vd.float()).cpu().numpy()
    u32, v32 = (x.float().double().cpu().numpy() for x in (ud, vd))
    assert _rel(jv, orc.jvp(u32, v32), fields) < 2e-5


@pytest.mark.parametrize("fields,n,batch", [(2, (5, 4, 4), 150), (3, (5, 4, 4), 150), (2, (49, 13, 13), 1)])
def test_three_elements_a_warp_equal_one(fields, n, batch):
    """FP64 at p = 1: many elements are taken three to a warp (the last ones fewer), few
    one to a warp. A batch of many against its points alone, bit for bit, and a large
    mesh against the oracle."""
    import torch
    import paper_2112_09271_gb300 as enp
    enp.build()
    P = _problem(1, fields, n)
    src = W.random_sources(P, 5)

    def values(u, v, b):
        op = enp.Operator(P, batch=b)
        op.set_sources(torch.tensor(src, device="cuda"), None)
        u, v = (torch.tensor(x, device="cuda") for x in (u, v))
        return [f.cpu().numpy().reshape(b, -1) for f in (op.residual(u), op.jvp(u, v), op.vjp(u, v))]

    us = [W.random_state(P, 1 + b % 4) for b in range(batch)]
    vs = [W.random_vector(P, 2 + b % 5) for b in range(batch)]
    many = values(np.concatenate(us), np.concatenate(vs), batch)
    if batch > 1:
        for b in (0, batch // 2, batch - 1):
            for x, y in zip(many, values(us[b], vs[b], 1)):
                np.testing.assert_array_equal(x[b], y[0])
        return
    orc = oracle.Oracle(P, src=src)
    ref = (orc.residual(us[0]), orc.jvp(us[0], vs[0]),
           orc.vjp_entries(us[0], vs[0], np.arange(P.n_dof)))
    for x, y in zip(many, ref):
        assert _rel(x[0], y, fields) < 1e-12
