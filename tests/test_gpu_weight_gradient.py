"""The weight-gradient kernel at the edges of its 32 x 4 x 2-point tiles: one tile, one point more or
less per axis, rows shorter than the three-point window, one point alone, more tiles than blocks.

Reference: the FP64 oracle, which rounds the layers' inputs to BF16 like the kernels.  An activation
can fall on the other side of a rounding boundary in FP32 (2^-8 of that value); the bounds of the
ordinary sizes (relative L2 1e-3, a layer's block 3e-3) leave room for that.  A tap, row or point
taken wrongly at an edge is several per cent at these sizes.
"""
import numpy as np
import pytest

import helm6_inputs as inputs
from oracle import cnn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(1, 1, 1, 1), (1, 2, 4, 2), (2, 1, 5, 3), (1, 3, 3, 31), (1, 2, 4, 32), (1, 3, 5, 33), (2, 2, 4, 66),
          (40, 5, 9, 35)]


@pytest.mark.parametrize("shape", SHAPES)
def test_weight_gradient_at_tile_edges(shape):
    from paper_1212_1397_gb300 import build, helm6
    build.build()
    th = cnn.init_params(inputs.standard_normal(21, cnn.n_params()))
    o = 0
    for ci, co in zip(cnn.CHANNELS[:-1], cnn.CHANNELS[1:]):
        o += co * ci * 27
        th[o:o + co] = 0.1 * inputs.standard_normal(22 + o, co)
        o += co
    th = th.astype(np.float32)
    n = int(np.prod(shape)) * 2
    x = inputs.standard_normal(23, n).reshape(shape + (2,)).astype(np.float32)
    t = inputs.standard_normal(24, n).reshape(shape + (2,)).astype(np.float32)
    with helm6.Trainer(*shape, th) as tr:
        _, g = tr.gradient(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
        _, g2 = tr.gradient(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    assert torch.equal(g, g2)
    g = g.cpu().numpy().astype(np.float64)
    _, ref = cnn.loss_and_grad(th.astype(np.float64), x.astype(np.float64), t.astype(np.float64), bf16=True)
    assert np.linalg.norm(g - ref) < 1e-3 * np.linalg.norm(ref)
    o = 0
    for ci, co in zip(cnn.CHANNELS[:-1], cnn.CHANNELS[1:]):
        for size in (co * ci * 27, co):
            b = slice(o, o + size)
            assert np.linalg.norm(g[b] - ref[b]) < 3e-3 * np.linalg.norm(ref[b]), (ci, co, size)
            o += size


@pytest.mark.parametrize("shape", [(1, 1, 130, 1), (2, 3, 64, 3), (1, 4, 9, 30), (2, 5, 31, 31), (1, 5, 8, 32),
                                   (1, 2, 3, 33), (2, 9, 32, 32)])
def test_forward_at_run_and_brick_edges(shape):
    """Layers at the edges of the convolution kernel's tiles: images up to 32 points wide are taken as
    runs of 128 points of rows joined by a zero point, wider ones as 30 x 4 x 4 bricks.  The bound is
    that of the ordinary sizes: FP32 sums and single BF16 rounding flips (2^-8 of a value)."""
    from paper_1212_1397_gb300 import build, helm6
    build.build()
    th = cnn.init_params(inputs.standard_normal(31, cnn.n_params())).astype(np.float32)
    x = inputs.standard_normal(32, int(np.prod(shape)) * 2).reshape(shape + (2,)).astype(np.float32)
    with helm6.Trainer(*shape, th) as tr:
        y = tr.forward(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    ref = cnn.forward(th.astype(np.float64), x.astype(np.float64), bf16=True)
    assert np.linalg.norm(y - ref) < 1e-3 * np.linalg.norm(ref)
    assert np.abs(y - ref).max() < 1e-2 * np.abs(ref).max()
