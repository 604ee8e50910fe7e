"""Hybrid Gauss-Seidel on levels large enough for a launch per colour, against its definition
x_i += (f - A x)_i / D_ii, colour after colour, with the library's residual and diagonal (which have
oracle tests of their own).  The macros share no node, so every skeleton node is a Dirichlet node and
keeps its value.  Tolerances as for the small levels in test_gpu_solvers.py."""

import numpy as np
import pytest

from paper_1908_08666_gb300 import binding as B

from hhg_gpu import Ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("macros,level", [(1, 5), (3, 6), (1, 7)])
def test_colours_follow_the_definition(macros, level):
    xyz = np.concatenate([np.vstack([np.zeros(3), np.eye(3)]) * (1 + 0.2 * m) + 3.0 * m for m in range(macros)])
    ctx = Ctx(xyz, np.arange(4 * macros).reshape(macros, 4), level, dict(nu=0.3))
    try:
        t = ctx.torch
        ctx.set_k(1.0 + 0.5 * np.sin(3.0 * ctx.coords_u[:, 0]) * np.cos(2.0 * ctx.coords_u[:, 1]))
        B.hhg_mg_setup(ctx.h)
        B.hhg_set_mg_params(ctx.h, smoother=B.SMOOTH_HYBRID_GS, omega=0.6, pre=1, post=1)
        n = 2**level
        ijk = np.array([(i, j, k) for k in range(n + 1) for j in range(n + 1 - k) for i in range(n + 1 - k - j)])
        inner = (ijk.min(axis=1) > 0) & (ijk.sum(axis=1) < n)
        col = np.where(inner, (ijk % 2) @ [4, 2, 1], -1)
        col = t.as_tensor(np.tile(col, 3 * macros), device="cuda")
        f = t.randn(3 * ctx.E, dtype=t.float64, device="cuda", generator=t.Generator("cuda").manual_seed(1))
        x0 = t.randn(3 * ctx.E, dtype=t.float64, device="cuda", generator=t.Generator("cuda").manual_seed(2))
        d, r, want = t.empty_like(f), t.empty_like(f), x0.clone()
        B.hhg_diagonal(ctx.h, level, B.F64, d)
        for c in range(8):
            B.hhg_residual(ctx.h, level, B.F64, f, want, r)
            want = t.where(col == c, want + r / d, want)
        scale = want.abs().max().item()
        for dt, tdt, tol in ((B.F64, t.float64, 1e-11), (B.F32, t.float32, 2e-5)):
            x = x0.to(tdt, copy=True)  # the sweep works in place
            B.hhg_smooth(ctx.h, level, dt, 1, f.to(tdt), x)
            t.cuda.synchronize()
            assert (x.double() - want).abs().max().item() <= tol * scale
            assert t.equal(x[col < 0], x0.to(tdt)[col < 0])
    finally:
        ctx.close()
