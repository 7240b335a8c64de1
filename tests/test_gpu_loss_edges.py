"""Eq. 3 loss at the edges of its tiles (32x54 output pixels, seven rows per thread, quads of four
columns): images that end on, one before and one after them, thinner than the window, and flat
or saturated fields, against the FP64 oracle.  Tolerances are those of test_gpu_loss."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2409_18122_gb300 import gs

from test_gpu_loss import _check_grad, _flat, _run, _ssim_part

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(32, 54)], [(31, 53), (33, 55)], [(64, 108), (65, 109)], [(4, 7), (5, 8), (3, 6)],
                                   [(1, 60), (60, 1), (1, 1)], [(36, 49), (28, 56), (97, 163)]])
def test_loss_and_gradient_at_tile_edges(sizes):
    loss, g_rgb, g_depth, ref, (rgbs, rrefs) = _run(sizes, gs.EQ3_WEIGHTS, seed=11 + len(sizes) + sizes[0][0])
    L, l1d, l1c, ss, gr, gd = ref
    np.testing.assert_allclose(loss, [L, l1d, l1c, ss], rtol=2e-5)
    _check_grad(g_rgb, gr, _ssim_part(rgbs, rrefs, sizes, 0.1))
    np.testing.assert_allclose(g_depth, np.concatenate([g.reshape(-1) for g in gd]), rtol=1e-6, atol=0)


@pytest.mark.parametrize("x,y", [(0.0, 0.0), (1.0, 1.0), (0.0, 1.0), (0.5, 0.25)])
def test_flat_images(x, y):
    """Constant images: the variances vanish and S is decided by C1 and C2."""
    W, H = 45, 70
    rgbs, rrefs = [np.full((3, H, W), x, np.float32)], [np.full((3, H, W), y, np.float32)]
    d = [np.full((H, W), 2.0, np.float32)]
    loss, _, _ = gs.ImageLoss([(W, H)])(_flat(rgbs), _flat(d), _flat(rrefs), _flat(d))
    torch.cuda.synchronize()
    L = O.mapping_loss_views(rgbs, d, rrefs, d, *gs.EQ3_WEIGHTS)[0]
    np.testing.assert_allclose(float(loss[0]), L, rtol=2e-5, atol=2e-6)


@pytest.mark.parametrize("h", [2, 6, 7, 8, 14, 43, 44, 45, 47, 49, 50, 61, 62, 108 + 43, 108 + 44])
def test_heights_that_end_inside_a_tile(h):
    """Only the input rows that some output row of the view takes are blurred (height of the last
    tile + 10, at most 64), seven output rows per warp: heights on both sides of each."""
    sizes = [(35, h), (70, h + 1)]
    loss, g_rgb, g_depth, ref, (rgbs, rrefs) = _run(sizes, gs.EQ3_WEIGHTS, seed=h)
    L, l1d, l1c, ss, gr, gd = ref
    np.testing.assert_allclose(loss, [L, l1d, l1c, ss], rtol=2e-5)
    _check_grad(g_rgb, gr, _ssim_part(rgbs, rrefs, sizes, 0.1))
    np.testing.assert_allclose(g_depth, np.concatenate([g.reshape(-1) for g in gd]), rtol=1e-6, atol=0)
