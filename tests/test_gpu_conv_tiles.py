"""The default network convolution and weight gradient at the edges of their tiles: rows that end inside
a group of four voxels, one group over a tile, planes that end inside a march, both tile forms.  Oracle
and tolerances as in test_gpu_learned.py."""

import numpy as np
import pytest

from oracle import learned as LN
from paper_1908_08666_gb300 import binding as B

from test_gpu_learned import _flat, _params, _unflat, ctx  # noqa: F401  (module fixture)

pytestmark = pytest.mark.gpu


# grids under and over the size (456 tiles of 4 x 4 x 32 voxels) from which the default is the grouped
# tcgen05 kernel
SMALL = [(1, 5, 16, 32), (1, 3, 17, 33), (2, 6, 33, 66), (1, 33, 20, 129), (1, 1, 11, 36)]
LARGE = [(1, 29, 65, 127), (1, 33, 65, 66), (2, 16, 129, 65), (1, 5, 160, 165), (8, 31, 31, 32), (1, 2, 256, 257)]


@pytest.mark.parametrize("shape", SMALL + LARGE)
def test_forward_at_tile_edges(ctx, shape):  # noqa: F811
    t = ctx.torch
    B.hhg_learn_set_conv_kernel(ctx.h, 0)
    Ws, bs = _params(4)
    B.hhg_learn_set_params(ctx.h, _flat(Ws, bs))
    x = np.random.default_rng(sum(shape)).normal(size=shape + (LN.CIN,)).astype(np.float32)
    out = t.empty(shape + (LN.COUT,), dtype=t.float32, device="cuda")
    B.hhg_learn_forward(ctx.h, ctx.dev(x, t.float32), LN.CIN, *shape, out, LN.COUT)
    t.cuda.synchronize()
    want, _ = LN.forward(x.astype(np.float64), Ws, bs, cout=LN.COUT)
    got = out.cpu().numpy().astype(np.float64)
    assert np.abs(got - want).max() <= 1e-2 * np.abs(want).max()
    assert np.linalg.norm(got - want) <= 3e-3 * np.linalg.norm(want)


@pytest.mark.parametrize("shape", SMALL[:3] + [(1, 29, 65, 127)])
def test_gradients_at_tile_edges(ctx, shape):  # noqa: F811
    t = ctx.torch
    B.hhg_learn_set_conv_kernel(ctx.h, 0)
    Ws, bs = _params(5)
    B.hhg_learn_set_params(ctx.h, _flat(Ws, bs))
    rng = np.random.default_rng(20 + sum(shape))
    x = rng.normal(size=shape + (LN.CIN,)).astype(np.float32)
    tgt = rng.normal(size=shape + (LN.COUT,)).astype(np.float32)
    loss, g = B.hhg_learn_loss_grad(ctx.h, ctx.dev(x, t.float32), LN.CIN, ctx.dev(tgt, t.float32), *shape, LN.COUT)
    wl, dWs, dbs = LN.loss_and_grads(x.astype(np.float64), tgt.astype(np.float64), Ws, bs, cout=LN.COUT)
    assert abs(loss - wl) <= 1e-3 * wl
    gW, gb = _unflat(g.astype(np.float64))
    for l in range(4):
        assert np.linalg.norm(gW[l] - dWs[l]) <= 2e-2 * np.linalg.norm(dWs[l]), l
        assert np.linalg.norm(gb[l] - dbs[l]) <= 2e-2 * np.linalg.norm(dbs[l]) + 1e-12, l


@pytest.mark.parametrize("shape", SMALL + LARGE)
def test_every_kernel_sums_in_the_same_order(ctx, shape):  # noqa: F811
    """A hidden activation is rounded to BF16, so another order of the sums shows in the outputs: the three
    kernels agree to the last bit."""
    t = ctx.torch
    Ws, bs = _params(6)
    B.hhg_learn_set_params(ctx.h, _flat(Ws, bs))
    x = ctx.dev(np.random.default_rng(sum(shape)).normal(size=shape + (LN.CIN,)), t.float32)
    outs = []
    try:
        for kernel in (0, 1, 2):
            B.hhg_learn_set_conv_kernel(ctx.h, kernel)
            outs.append(t.empty(shape + (LN.COUT,), dtype=t.float32, device="cuda"))
            B.hhg_learn_forward(ctx.h, x, LN.CIN, *shape, outs[-1], LN.COUT)
        t.cuda.synchronize()
    finally:
        B.hhg_learn_set_conv_kernel(ctx.h, 0)
    assert t.equal(outs[0], outs[1]) and t.equal(outs[0], outs[2])
