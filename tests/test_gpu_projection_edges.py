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


def _check_visible(gmap, cams, prm):
    n = gmap.n
    fr = gs.Frame(n, cams, prm)
    fr.project(gs.GaussianMapTensors.from_numpy(gmap))
    torch.cuda.synchronize()
    rec = gpu_records(fr)
    vis = O.project(gmap, cams, oparams(prm))["vis"].astype(bool)
    n_grp = (n + 31) // 32
    masks = rec["grp_mask"].reshape(len(cams), n_grp)
    got = ((masks[:, :, None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(len(cams), -1)[:, :n].astype(bool)
    np.testing.assert_array_equal(got, vis)
    return vis


@pytest.mark.parametrize("scale", [0.25, 1.5, 6.0])
def test_visible_sets_of_scaled_and_sheared_cameras(scale):
    """R is used as it is given: lengths in the camera's frame are those of R^T, also where R is not
    a rotation (a pose with a scale, a shear), so the culls that bound them must follow it."""
    gmap = _map(20_011, 7)
    shear = np.array([[1.0, 0.4, -0.2], [0.0, 1.0, 0.3], [0.0, 0.1, 1.0]])
    cams = [Camera(97.0, 97.0, 48.5, 30.5, 97, 61, (scale * m).astype(np.float32), np.zeros(3, np.float32))
            for m in (np.eye(3), shear, np.diag([1.0, 1.0, 1.0 / scale]), np.diag([1.0 / scale, 1.0, 1.0]))]
    vis = _check_visible(gmap, cams, gs.RenderParams())
    assert vis[:2].sum(axis=1).min() > 1000


def test_visible_sets_with_a_far_principal_point():
    """A guard band of 1e5 and an image four million pixels off the optical axis: the means are
    rounded to quarters of a pixel, of which the half-pixel supports are not independent."""
    rng = np.random.default_rng(5)
    n = 20_011
    tz = rng.uniform(20.0, 60.0, n)
    px = np.where(rng.random(n) < 0.5, rng.uniform(-1.5, 1.5, n), 97.0 + rng.uniform(-1.5, 1.5, n))
    mo = np.stack([(px + 4.0e6) / 100.0 * tz, rng.uniform(-0.25, 0.25, n) * tz, tz, rng.uniform(-5.05, -4.9, n)], 1)
    q = rng.standard_normal((n, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    su = np.full((n, 4), -13.0)
    gmap = GaussianMap(*(a.astype(np.float32) for a in (mo, su, q, np.zeros((n, 4)))))
    cam = Camera(100.0, 100.0, -4.0e6, 30.5, 97, 61, np.eye(3, dtype=np.float32), np.zeros(3, np.float32))
    vis = _check_visible(gmap, [cam], gs.RenderParams(guard=1.0e5))
    assert 0.05 < vis.mean() < 0.95
