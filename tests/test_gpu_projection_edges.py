"""The projection's visibility where its shortcuts end: means within a few pixels of the image's
borders, opacities at the floor, scales from specks to larger than the room, needles, means near
the near plane, principal points outside the image, one-pixel images, low-pass 0 and large, no
opacity floor.  Visible sets and record counts are the oracle's exactly."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2409_18122_gb300 import gs
from paper_2409_18122_gb300.scenes import Camera, GaussianMap

from gpu_helpers import gpu_records
from test_gpu_parity import oparams

pytestmark = pytest.mark.gpu


def _map(n, seed):
    rng = np.random.default_rng(seed)
    tz = np.exp(rng.uniform(np.log(0.15), np.log(60.0), n))
    side = rng.choice([-1.0, 1.0], (n, 2)) * (0.5 + rng.choice([0.0, 0.01, 0.05, 0.2], (n, 2)) * rng.standard_normal((n, 2)))
    side[rng.random(n) < 0.3] = rng.uniform(-0.7, 0.7, 2)      # x / tz in widths: borders at +-0.5
    mo = np.stack([side[:, 0] * tz, side[:, 1] * 0.7 * tz, tz, rng.choice([-5.6, -5.53, -4.0, 0.0, 6.0], n)], 1)
    ls = rng.choice([-9.0, -5.0, -3.0, 0.0, 3.5], (n, 1)) + rng.choice([0.0, 0.5, 4.0], (n, 1)) * rng.standard_normal((n, 3))
    q = rng.standard_normal((n, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    su = np.concatenate([np.clip(ls, -20, 6), rng.uniform(0, 1, (n, 1))], 1)
    f32 = lambda a: a.astype(np.float32)  # noqa: E731
    return GaussianMap(f32(mo), f32(su), f32(q), np.zeros((n, 4), np.float32))


@pytest.mark.parametrize("eps2d,alpha_min", [(0.3, 1.0 / 255.0), (0.0, 1.0 / 255.0), (5.0, 0.02), (0.3, 0.0), (1e-3, 1e-4)])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_visible_sets(seed, eps2d, alpha_min):
    n = 20_011
    gmap = _map(n, seed)
    eye, zero = np.eye(3, dtype=np.float32), np.zeros(3, np.float32)
    cams = [Camera(97.0, 97.0, 48.5, 30.5, 97, 61, eye, zero), Camera(640.0, 640.0, 320.0, 224.0, 640, 448, eye, zero),
            Camera(33.0, 35.0, -70.0, 9.0, 33, 21, eye, zero), Camera(2.0, 2.0, 0.5, 0.5, 1, 1, eye, zero),
            Camera(2000.0, 900.0, 1000.0, 3.0, 2001, 7, eye, zero)]
    prm = gs.RenderParams(eps2d=eps2d, alpha_min=alpha_min)
    fr = gs.Frame(n, cams, prm)
    fr.project(gs.GaussianMapTensors.from_numpy(gmap))
    torch.cuda.synchronize()
    rec = gpu_records(fr)
    vis = O.project(gmap, cams, oparams(prm))["vis"].astype(bool)
    n_grp = (n + 31) // 32
    bits = np.zeros((n_grp * 32, len(cams)), bool)
    bits[:n] = vis.T
    masks = (bits.reshape(n_grp, 32, len(cams)) * (1 << np.arange(32, dtype=np.uint64))[None, :, None]).sum(axis=1)
    np.testing.assert_array_equal(rec["grp_mask"].reshape(len(cams), n_grp), masks.astype(np.uint32).T)
    assert rec["n"] == int(vis.sum()) and 0 < rec["n"] < n * len(cams)
    # every counted record was written by the write pass: ids in order, per view the visible ones
    for v in range(len(cams)):
        np.testing.assert_array_equal(rec["gid"][rec["view"] == v], np.flatnonzero(vis[v]))
