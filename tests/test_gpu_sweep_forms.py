"""The one-launch sweep where its layout changes with the level: macros of few columns that share a block, faces
and edges of few nodes, columns of one, two and more points in FP64 and of more than two in FP32.  Against
the interior kernels of hhg_set_interior_kernel (which share the skeleton rows), and on coarse levels
against the oracle.

Tolerances.  FP64: two sums of the same terms, 1e-11 of the largest value as in test_gpu_rows.py.  FP32: the
rounding bound of test_gpu_parity.py is 64 2^-24 sum_j |A_ij| |x_j - x_i|; for random x the 42 terms of a row
sum to at most sqrt(42) < 10 times their root mean square, and the largest |A x| of many rows is at least
that; twice the bound, since both sides round."""

import numpy as np
import pytest

import hhg_inputs as hi
from oracle import mesh, operators as op
from paper_1908_08666_gb300 import binding as B

from hhg_gpu import Ctx
from test_gpu_parity import FP32_C, _fp32_scale, _kfun, _oracle

pytestmark = pytest.mark.gpu

F64, F32 = 1e-11, 2 * 10 * FP32_C


def _box162():
    return hi.kuhn_box(3, 3, 3)


def _close(got, want, comps, tol):
    for g, w in zip(got.double().reshape(comps, -1), want.double().reshape(comps, -1)):
        assert (g - w).abs().max().item() <= tol * w.abs().max().item()


def _sweeps(ctx, comps, dt, tdt, tol, kernels):
    """apply, residual and its norm of kernel 0 against the others'"""
    t, l = ctx.torch, ctx.level
    x = ctx.to_lib(hi.node_noise(ctx.coords_u, seed=3, comps=comps), tdt, comps)
    f = ctx.to_lib(hi.node_noise(ctx.coords_u, seed=4, comps=comps), tdt, comps)
    ap, re = (B.hhg_apply, B.hhg_residual) if comps == 3 else (B.hhg_stokes_apply, B.hhg_stokes_residual)
    out = []
    for kernel in kernels:
        B.hhg_set_interior_kernel(ctx.h, kernel)
        y, r = t.full_like(x, 7.0), t.full_like(x, 7.0)
        ap(ctx.h, l, dt, x, y)
        out.append((y, r, re(ctx.h, l, dt, f, x, r, want_norm=True)))
    B.hhg_set_interior_kernel(ctx.h, 0)
    for y, r, norm2 in out[1:]:
        _close(out[0][0], y, comps, tol)
        _close(out[0][1], r, comps, tol)
        assert abs(out[0][2] - norm2) <= 2 * tol * norm2
    return x, f


@pytest.mark.parametrize("builder,level", [(hi.kuhn_cube, 2), (hi.kuhn_cube, 3), (hi.unit_tet, 2), (_box162, 2),
                                           (_box162, 3), (hi.unit_tet, 4), (hi.unit_tet, 7)],
                         ids=["cube_l2", "cube_l3", "one_l2", "box_l2", "box_l3", "one_l4", "one_l7"])
@pytest.mark.parametrize("problem", [{}, dict(khat=B.KHAT_EDGE), dict(kind=B.STOKES)],
                         ids=["elasticity", "edge", "stokes"])
def test_sweeps_equal_interior_kernels(builder, level, problem):
    ctx = Ctx(*builder(), level, problem)
    try:
        ctx.set_k(_kfun(ctx.coords_u))
        comps = 4 if "kind" in problem else 3
        for dt, tdt, tol in ((B.F64, ctx.torch.float64, F64), (B.F32, ctx.torch.float32, F32)):
            _sweeps(ctx, comps, dt, tdt, tol, (0, 3))
    finally:
        ctx.close()


@pytest.mark.parametrize("count,level", [(2, 2), (3, 2)])
def test_coarse_rows_match_oracle(count, level):
    """Faces and edges of three nodes, on 48 and on 162 macros."""
    xyz, tets = hi.kuhn_cube(count)
    mm, lv, A = _oracle(xyz, tets, level, _kfun)
    ctx = Ctx(xyz, tets, level, dict(nu=0.3))
    try:
        t = ctx.torch
        perm = mesh.match_nodes(lv.coords, ctx.coords_u)
        ctx.set_k(_kfun(ctx.coords_u))
        x_or = hi.node_noise(lv.coords, seed=7)
        x_u = np.empty_like(x_or)
        x_u[perm] = x_or
        y_or = op.apply(op.with_dirichlet_rows(A, lv.dirichlet), x_or)
        scale, free = _fp32_scale(A, x_or, lv), ~lv.dirichlet
        for dt, tdt in ((B.F64, t.float64), (B.F32, t.float32)):
            x = ctx.to_lib(x_u, tdt, 3)
            y = t.full_like(x, 7.0)
            B.hhg_apply(ctx.h, level, dt, x, y)
            yg = ctx.from_lib(y, 3)
            assert np.array_equal(y.double().cpu().numpy().reshape(3, ctx.E).T, yg[ctx.e2u])
            if dt == B.F64:
                assert np.abs(yg[perm] - y_or).max() <= 1e-12 * np.abs(y_or).max()
            else:
                assert np.all(np.abs(yg[perm] - y_or)[free] <= FP32_C * scale[free] + 1e-30)
    finally:
        ctx.close()


@pytest.mark.parametrize("problem", [{}, dict(khat=B.KHAT_EDGE), dict(variant=B.UNPHYSICAL), dict(kind=B.STOKES)],
                         ids=["elasticity", "edge", "unphysical", "stokes"])
def test_long_columns(problem):
    """129^3 nodes: columns of four points in FP32 and two in FP64, every epilogue."""
    ctx = Ctx(*hi.kuhn_cube(), 7, problem)
    try:
        t = ctx.torch
        ctx.set_k(_kfun(ctx.coords_u))
        comps = 4 if "kind" in problem else 3
        for dt, tdt, tol in ((B.F64, t.float64, F64), (B.F32, t.float32, F32)):
            x, f = _sweeps(ctx, comps, dt, tdt, tol, (0, 3))
            if comps == 4:
                continue
            B.hhg_mg_setup(ctx.h)
            d = []
            for kernel in (0, 3):
                B.hhg_set_interior_kernel(ctx.h, kernel)
                d.append(t.full_like(x, 7.0))
                B.hhg_diagonal(ctx.h, 7, dt, d[-1])
            _close(d[0], d[1], 3, tol)
            for smoother in (B.SMOOTH_CHEBYSHEV, B.SMOOTH_JACOBI):
                B.hhg_set_mg_params(ctx.h, smoother=smoother)
                out = []
                for kernel in (0, 3):
                    B.hhg_set_interior_kernel(ctx.h, kernel)
                    out.append(x.clone())
                    B.hhg_smooth(ctx.h, 7, dt, 2, f * 1e-3, out[-1])
                t.cuda.synchronize()
                _close(out[0], out[1], 3, tol)
    finally:
        ctx.close()


def test_long_columns_bf16_coefficient():
    ctx = Ctx(*hi.kuhn_cube(), 7, dict(nu=0.3))
    try:
        t = ctx.torch
        k = ctx.to_lib(_kfun(ctx.coords_u), t.float64, 1)
        B.hhg_set_coefficient(ctx.h, k.to(t.bfloat16), B.BF16)
        _sweeps(ctx, 3, B.F32, t.float32, F32, (0, 3))
    finally:
        ctx.close()


def test_columns_of_four_points_in_fp64():
    ctx = Ctx(*hi.skewed_pair(), 8, dict(nu=0.3))
    try:
        ctx.set_k(_kfun(ctx.coords_u))
        _sweeps(ctx, 3, B.F64, ctx.torch.float64, F64, (0, 3))
    finally:
        ctx.close()


@pytest.mark.parametrize("builder,level,problem", [(_box162, 2, {}), (_box162, 3, {}), (hi.unit_tet, 2, {}),
                                                   (hi.skewed_pair, 4, dict(variant=B.STORED)), (hi.kuhn_cube, 7, {})],
                         ids=["box_l2", "box_l3", "one_l2", "pair_stored", "cube_l7"])
def test_noalloc_residual(builder, level, problem):
    """The residual without allocation against hhg_residual, up to the largest levels that its scratch takes;
    tolerances of test_zz_no_alloc.py."""
    ctx = Ctx(*builder(), level, dict(nu=0.3, **problem))
    try:
        t = ctx.torch
        ctx.set_k(_kfun(ctx.coords_u))
        for dt, tdt, tol in ((B.F64, t.float64, 1e-12), (B.F32, t.float32, FP32_C)):
            x = ctx.to_lib(hi.node_noise(ctx.coords_u, seed=3), tdt, 3)
            f = ctx.to_lib(hi.node_noise(ctx.coords_u, seed=4), tdt, 3)
            want, got = t.empty_like(x), t.full_like(x, float("nan"))
            n_want = B.hhg_residual(ctx.h, level, dt, f, x, want, want_norm=True)
            n_got = B.hhg_residual_noalloc(ctx.h, level, dt, f, x, got)
            t.cuda.synchronize()
            _close(got, want, 3, tol)
            assert abs(n_got - n_want) <= (1e-12 if dt == B.F64 else 1e-5) * n_want
    finally:
        ctx.close()
