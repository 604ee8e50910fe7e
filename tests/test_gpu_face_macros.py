"""Macro faces held by more than two macros.  The macro mesh is not checked for them, and the rows of such a
face's nodes are sums over all of its macros as anywhere else.  Oracle and tolerances as in
test_gpu_parity.py and test_gpu_stokes.py."""

import numpy as np
import pytest

import hhg_inputs as hi
from oracle import mesh, operators as op, stokes as ST
from paper_1908_08666_gb300 import binding as B

from hhg_gpu import Ctx
from test_gpu_parity import FP32_C, _fp32_scale, _kfun, _oracle

pytestmark = pytest.mark.gpu


def _book(count):
    """`count` macros on one face, their fourth vertices on both sides of it; the vertices' order differs
    from macro to macro, so that every kind of face occurs."""
    apex = np.random.default_rng(count).uniform(0.2, 1.0, (count, 3)) * [1, 1, 0.7]
    apex[::2, 2] *= -1
    xyz = np.concatenate([[[0.0, 0.0, 0.0], [1.0, 0.1, 0.0], [0.2, 1.0, 0.05]], apex])
    tets = [np.roll([0, 1, 2, 3 + q], q) for q in range(count)]
    return xyz, np.array(tets, dtype=np.int64)


@pytest.mark.parametrize("count,level", [(3, 2), (3, 4), (4, 3), (11, 3), (18, 2)])
def test_rows_of_a_face_in_many_macros(count, level):
    xyz, tets = _book(count)
    mm, lv, A = _oracle(xyz, tets, level, _kfun)
    ctx = Ctx(xyz, tets, level, dict(nu=0.3))
    try:
        t = ctx.torch
        perm = mesh.match_nodes(lv.coords, ctx.coords_u)
        ctx.set_k(_kfun(ctx.coords_u))
        x_or, f_or = hi.node_noise(lv.coords, seed=7), hi.node_noise(lv.coords, seed=8)
        x_u, f_u = np.empty_like(x_or), np.empty_like(f_or)
        x_u[perm], f_u[perm] = x_or, f_or
        y_or = op.apply(op.with_dirichlet_rows(A, lv.dirichlet), x_or)
        r_or = op.residual(A, f_or, x_or, lv.dirichlet)
        scale = _fp32_scale(A, x_or, lv)
        free = ~lv.dirichlet
        for kernel in (0, 2, 3):
            B.hhg_set_interior_kernel(ctx.h, kernel)
            for dt, tdt in ((B.F64, t.float64), (B.F32, t.float32)):
                x, f = ctx.to_lib(x_u, tdt, 3), ctx.to_lib(f_u, tdt, 3)
                y, r = t.full_like(x, 7.0), t.full_like(x, 7.0)
                B.hhg_apply(ctx.h, level, dt, x, y)
                norm2 = B.hhg_residual(ctx.h, level, dt, f, x, r, want_norm=True)
                yg, rg = ctx.from_lib(y, 3)[perm], ctx.from_lib(r, 3)[perm]
                if dt == B.F64:
                    assert np.abs(yg - y_or).max() <= 1e-12 * np.abs(y_or).max()
                    assert np.abs(rg - r_or).max() <= 1e-12 * np.abs(y_or).max()
                    assert abs(norm2 - (r_or[free] ** 2).sum()) <= 1e-11 * (r_or[free] ** 2).sum()
                else:
                    assert np.all(np.abs(yg - y_or)[free] <= FP32_C * scale[free] + 1e-30)
                for v in (y, r):  # every copy
                    full = v.double().cpu().numpy().reshape(3, ctx.E).T
                    assert np.array_equal(full, ctx.from_lib(v, 3)[ctx.e2u])
    finally:
        ctx.close()


def test_stokes_rows_of_a_face_in_many_macros():
    xyz, tets = _book(5)
    level = 3
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
        y = t.full_like(x, 7.0)
        B.hhg_stokes_apply(ctx.h, level, B.F64, x, y)
        yg = ctx.from_lib(y, 4)
        assert np.abs(ST.pack(yg[perm, :3], yg[perm, 3]) - y_or).max() <= 1e-12 * np.abs(y_or).max()
        assert np.array_equal(y.cpu().numpy().reshape(4, ctx.E).T, yg[ctx.e2u])
    finally:
        ctx.close()
