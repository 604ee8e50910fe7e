"""The Carreau viscosity on meshes of more macros than one launch takes, and with one interior node per
macro.  Oracle and tolerance as in test_gpu_carreau.py."""

import numpy as np
import pytest

from oracle import carreau as CA, mesh
from paper_1908_08666_gb300 import binding as B

from hhg_gpu import Ctx
from test_gpu_carreau import PAR, _u
from test_gpu_rows import _fan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,level", [(16, 2), (17, 3), (33, 2)])
def test_viscosity_over_several_launches(count, level):
    xyz, tets = _fan(count)
    lv = mesh.build_level(mesh.MacroMesh.build(xyz, tets), level)
    ctx = Ctx(xyz, tets, level, dict(kind=B.STOKES))
    try:
        t = ctx.torch
        perm = mesh.match_nodes(lv.coords, ctx.coords_u)
        mu = t.empty(ctx.E, dtype=t.float64, device="cuda")
        u = ctx.to_lib(_u(ctx.coords_u), t.float64, 3)
        B.hhg_carreau_viscosity(ctx.h, level, u, mu, **PAR)
        want = CA.viscosity(lv, _u(lv.coords), **PAR)
        assert np.abs(ctx.from_lib(mu, 1)[perm, 0] - want).max() <= 1e-11 * np.abs(want).max()
        # a velocity that is not finite at an interior node makes that node's viscosity not finite
        n = 2**level
        ijk = np.array([(i, j, k) for k in range(n + 1) for j in range(n + 1 - k) for i in range(n + 1 - k - j)])
        e = int(np.nonzero((ijk == 1).all(axis=1))[0][0]) + (count - 1) * len(ijk)
        u[e] = float("nan")
        B.hhg_carreau_viscosity(ctx.h, level, u, mu, **PAR)
        assert t.isnan(mu[e]).item()
    finally:
        ctx.close()
