"""The skeleton-row kernel where its lane layout changes: nodes in more macros than a warp has lanes,
faces without a macro-interior neighbour, levels on both sides of the size up to which it sweeps all
nodes.  Oracle and tolerances as in test_gpu_parity.py and test_gpu_stokes.py."""

import numpy as np
import pytest

import hhg_inputs as hi
from oracle import mesh, operators as op, stokes as ST
from paper_1908_08666_gb300 import binding as B

from hhg_gpu import Ctx
from test_gpu_parity import FP32_C, _fp32_scale, _kfun, _oracle

pytestmark = pytest.mark.gpu


def _fan(count):
    """`count` macros around one interior edge."""
    a = 2 * np.pi * np.arange(count) / count
    ring = np.stack([np.cos(a), np.sin(a), 0.5 + 0.2 * np.cos(3 * a)], axis=1)
    xyz = np.concatenate([[[0.0, 0.0, 0.0], [0.0, 0.0, 1.0]], ring])
    tets = [[0, 1, 2 + q, 2 + (q + 1) % count] for q in range(count)]
    return xyz, np.array(tets, dtype=np.int64)


def _fan_neumann(count):
    """The fan with free outer faces around vertex 0 (the faces that do not hold vertex 1)."""
    xyz, tets = _fan(count)
    flags = np.ones((count, 4), dtype=np.int32)
    flags[:, 1] = 0
    return xyz, tets, flags


@pytest.mark.parametrize("count,level", [(33, 2), (36, 3), (65, 2), (8, 3)])
def test_nodes_in_many_macros(count, level):
    xyz, tets = _fan(count)
    mm, lv, A = _oracle(xyz, tets, level, _kfun)
    A_bc = op.with_dirichlet_rows(A, lv.dirichlet)
    ctx = Ctx(xyz, tets, level, dict(nu=0.3))
    try:
        t = ctx.torch
        perm = mesh.match_nodes(lv.coords, ctx.coords_u)
        ctx.set_k(_kfun(ctx.coords_u))
        x_or = hi.node_noise(lv.coords, seed=7)
        x_u = np.empty_like(x_or)
        x_u[perm] = x_or
        y_or = op.apply(A_bc, x_or)
        scale = _fp32_scale(A, x_or, lv)
        for kernel in (0, 2, 3):
            B.hhg_set_interior_kernel(ctx.h, kernel)
            for dt, tdt in ((B.F64, t.float64), (B.F32, t.float32)):
                x = ctx.to_lib(x_u, tdt, 3)
                y = t.empty_like(x)
                B.hhg_apply(ctx.h, level, dt, x, y)
                yg = ctx.from_lib(y, 3)[perm]
                if dt == B.F64:
                    assert np.abs(yg - y_or).max() <= 1e-12 * np.abs(y_or).max()
                else:
                    free = ~lv.dirichlet
                    assert np.all(np.abs(yg - y_or)[free] <= FP32_C * scale[free] + 1e-30)
                full = y.double().cpu().numpy().reshape(3, ctx.E).T
                assert np.array_equal(full, ctx.from_lib(y, 3)[ctx.e2u])
    finally:
        ctx.close()


def test_stokes_rows_of_nodes_in_many_macros():
    xyz, tets = _fan(34)
    level = 2
    mm = mesh.MacroMesh.build(xyz, tets)
    lv = mesh.build_level(mm, level)
    Kbc, _ = ST.stokes_operator(mm, lv, _kfun(lv.coords))
    ctx = Ctx(xyz, tets, level, dict(kind=B.STOKES))
    try:
        t = ctx.torch
        perm = mesh.match_nodes(lv.coords, ctx.coords_u)
        ctx.set_k(_kfun(ctx.coords_u))
        xu, xp = hi.node_noise(lv.coords, 5), hi.node_noise(lv.coords, 6, comps=1)
        y_or = Kbc @ ST.pack(xu, xp)
        x_u = np.empty((lv.num_nodes, 4))
        x_u[perm, :3], x_u[perm, 3] = xu, xp
        x = ctx.to_lib(x_u, t.float64, 4)
        y = t.empty_like(x)
        B.hhg_stokes_apply(ctx.h, level, B.F64, x, y)
        yg = ctx.from_lib(y, 4)[perm]
        assert np.abs(ST.pack(yg[:, :3], yg[:, 3]) - y_or).max() <= 1e-12 * np.abs(y_or).max()
    finally:
        ctx.close()


def test_free_boundary_faces():
    """Free nodes with one incidence (outer faces) and a free vertex in every macro."""
    xyz, tets, flags = _fan_neumann(34)
    level = 2
    ctx = Ctx(xyz, tets, level, dict(nu=0.3), dirichlet_face_flags=flags)
    try:
        t = ctx.torch
        lv = mesh.build_level(mesh.MacroMesh.build(xyz, tets, flags), level)
        mm, _, A = _oracle(xyz, tets, level, _kfun)
        perm = mesh.match_nodes(lv.coords, ctx.coords_u)
        assert np.array_equal(ctx.udir[perm], lv.dirichlet)
        ctx.set_k(_kfun(ctx.coords_u))
        x_or = hi.node_noise(lv.coords, seed=7)
        x_u = np.empty_like(x_or)
        x_u[perm] = x_or
        y_or = op.apply(op.with_dirichlet_rows(A, lv.dirichlet), x_or)
        x = ctx.to_lib(x_u, t.float64, 3)
        y = t.empty_like(x)
        B.hhg_apply(ctx.h, level, B.F64, x, y)
        assert np.abs(ctx.from_lib(y, 3)[perm] - y_or).max() <= 1e-12 * np.abs(y_or).max()
    finally:
        ctx.close()


@pytest.mark.parametrize("builder,level", [(hi.unit_tet, 4), (hi.unit_tet, 5), (hi.unit_tet, 6), (hi.skewed_pair, 5)],
                         ids=["one_l4", "one_l5", "one_l6", "pair_l5"])
def test_all_rows_equal_interior_kernels(builder, level):
    """One launch over all nodes against the interior kernels, on sizes on both sides of its limit:
    every smoother epilogue runs in the V-cycle, both are FP64 sums of the same terms."""
    xyz, tets = builder()
    ctx = Ctx(xyz, tets, level, dict(nu=0.3))
    try:
        t = ctx.torch
        ctx.set_k(_kfun(ctx.coords_u))
        B.hhg_mg_setup(ctx.h)
        free = (~ctx.udir)[:, None]
        x_u = hi.node_noise(ctx.coords_u, seed=3) * free
        f = ctx.to_lib(hi.node_noise(ctx.coords_u, seed=4) * free, t.float64, 3)
        out = []
        for kernel in (0, 2, 3):
            B.hhg_set_interior_kernel(ctx.h, kernel)
            for smoother in (B.SMOOTH_CHEBYSHEV, B.SMOOTH_JACOBI):
                B.hhg_set_mg_params(ctx.h, smoother=smoother)
                B.hhg_mg_setup(ctx.h)
                x = ctx.to_lib(x_u, t.float64, 3)
                B.hhg_vcycle(ctx.h, level, B.F64, f, x)
                out.append(ctx.from_lib(x, 3))
        for q in range(2, 6):
            assert np.abs(out[q] - out[q % 2]).max() <= 1e-11 * np.abs(out[q % 2]).max()
    finally:
        ctx.close()
