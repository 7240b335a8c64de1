"""Backward compositing at the edges of its batches: lists of 0, 1, 15, 16, 17, 31, 32, 33 and
100 overlapping entries per pixel block (entries are summed sixteen at a time, groups of 32
list entries), ragged images, entries hidden behind saturated pixels, gradients of colour
only, depth only or both.  Reference: the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2409_18122_gb300 import gs, scenes

pytestmark = pytest.mark.gpu


def _stack(n, opaque, seed):
    """n Gaussians one behind the other, all covering the small image."""
    rng = np.random.default_rng(seed)
    mu = np.stack([rng.normal(0, 0.1, n), rng.normal(0, 0.1, n), np.linspace(2.0, 4.0, n)], 1) if n else np.zeros((0, 3))
    ls = rng.normal(-0.7, 0.2, (n, 3))
    q = rng.normal(size=(n, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    logit = rng.normal(2.5 if opaque else -3.0, 0.3, n)
    return scenes._pack(mu, ls, q, logit, rng.uniform(0, 1, (n, 3)), rng.uniform(0, 1, n))


@pytest.mark.parametrize("opaque", [False, True])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 100])
@pytest.mark.parametrize("which", ["both", "rgb", "depth"])
def test_gradients_of_stacked_entries(n, opaque, which):
    g = _stack(n, opaque, 40 + n)
    cam = scenes.Camera(40.0, 40.0, 9.5, 6.5, 19, 13)   # ragged: the image ends inside its blocks
    gm = gs.GaussianMapTensors.from_numpy(g)
    fr = gs.Frame(n, [cam])
    img = fr.forward(gm)
    ref = O.render_images(g, [cam])[0]
    rng = np.random.default_rng(n)
    d = rng.normal(size=(13, 19, 4))
    d[ref["knife"]] = 0.0                               # skip / stop decisions within rounding
    if which == "rgb":
        d[..., 3] = 0.0
    if which == "depth":
        d[..., :3] = 0.0
    d_rgb = None if which == "depth" else torch.from_numpy(
        np.ascontiguousarray(d[..., :3].transpose(2, 0, 1)).reshape(-1)).float().cuda()
    d_dep = None if which == "rgb" else torch.from_numpy(np.ascontiguousarray(d[..., 3]).reshape(-1)).float().cuda()
    out = fr.render_bwd(gm, img, d_rgb, d_dep)
    gref = O.grad(g, [cam], [d])
    for k in ("dmo", "dsu", "dq", "drgb"):
        a, b = out[k].cpu().numpy().astype(np.float64), gref[k]
        # FP32 replay through up to n layers: T is divided back n times (n 2^-24), and the sums
        # over the pixels cancel to within the rounding of their largest terms
        tol = 2e-3 * np.abs(b).max() + 1e-7
        np.testing.assert_allclose(a, b, rtol=0, atol=tol, err_msg=k)
