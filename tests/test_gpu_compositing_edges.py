"""Forward and information-gain compositing at the edges of its staging: lists whose length
ends inside a chunk, a group of 32 or the 64-entry ring, pixels that saturate in the middle of
a chunk or never, and alpha_min = 0 (no entry is skipped, the padding of a list's last chunk
must still add nothing), against the oracle.  Tolerances are gpu_helpers'."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2409_18122_gb300 import gs
from paper_2409_18122_gb300.scenes import Camera, GaussianMap

from gpu_helpers import DEPTH_RTOL, GRAD_RTOL, IG_RTOL, IMG_ATOL, images_host

pytestmark = pytest.mark.gpu


def _stack(n, logit, seed=0):
    """n Gaussians of about 2 to 6 pixels one behind another in front of an odd-sized 13 x 9 view."""
    rng = np.random.default_rng(seed + n)
    mo = np.zeros((n, 4), np.float32)
    mo[:, :2] = rng.uniform(-0.5, 0.5, (n, 2))
    mo[:, 2] = 2.0 + np.arange(n) * 0.01
    mo[:, 3] = logit + 0.3 * rng.standard_normal(n)
    su = np.concatenate([rng.uniform(-2.0, -1.0, (n, 3)), rng.uniform(0, 1, (n, 1))], 1).astype(np.float32)
    q = rng.standard_normal((n, 4))
    q = (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)
    rgb = np.concatenate([rng.uniform(0, 1, (n, 3)), np.zeros((n, 1))], 1).astype(np.float32)
    cam = Camera(30.0, 30.0, 6.5, 4.5, 13, 9, np.eye(3, dtype=np.float32), np.zeros(3, np.float32))
    return GaussianMap(mo, su, q, rgb), [cam]


@pytest.mark.parametrize("logit", [-4.0, 0.0])      # transparent: nothing saturates; opaque: all lanes do
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 63, 64, 65, 97])
def test_list_lengths(n, logit):
    gmap, cams = _stack(n, logit)
    gm = gs.GaussianMapTensors.from_numpy(gmap)
    ref = O.render_images(gmap, cams)[0]
    outs = []
    for b in gs.FWD_BATCH_CANDIDATES:
        fr = gs.Frame(n, cams, gs.RenderParams(fwd_batch=b))
        img = fr.forward(gm, fr.new_images(with_counts=True))
        torch.cuda.synchronize()
        fr.check_status()
        h = images_host(fr, img)[0]
        h["n_contrib"] = img["n_contrib"].cpu().numpy()
        outs.append(h)
        ok = ~ref["knife"]                    # pixels whose skip and stop decisions are clear of rounding
        for k in ("rgb", "unc", "T"):
            np.testing.assert_allclose(h[k][ok], ref[k][ok], rtol=0, atol=IMG_ATOL, err_msg=k)
        np.testing.assert_allclose(h["depth"][ok], ref["depth"][ok], rtol=0, atol=DEPTH_RTOL * (2.0 + 0.01 * n))
    for o in outs[1:]:
        for k in ("rgb", "depth", "unc", "T", "last", "n_contrib"):
            np.testing.assert_array_equal(o[k], outs[0][k])
    if not ref["knife"].any():
        for b in gs.IG_BATCH_CANDIDATES:
            ig = float(gs.InfoGain(n, cams, gs.RenderParams(ig_batch=b))(gm)[0])
            assert abs(ig - ref["unc"].mean()) <= IG_RTOL * abs(ref["unc"].mean()) + 1e-7


@pytest.mark.parametrize("n", [1, 3, 5, 33])
def test_padding_adds_nothing_without_an_opacity_floor(n):
    """alpha_min = 0: the padded entries of the last chunk (alpha = 0) are not skipped by the
    floor; colours that were staged by earlier work (here infinite ones) must not leak in."""
    gmap, cams = _stack(n, -1.0)
    hot = GaussianMap(gmap.mo, gmap.su, gmap.q, np.full_like(gmap.rgb, np.inf))
    prm = gs.RenderParams(alpha_min=0.0)
    gs.Frame(n, cams, prm).forward(gs.GaussianMapTensors.from_numpy(hot))
    fr = gs.Frame(n, cams, prm)
    img = fr.forward(gs.GaussianMapTensors.from_numpy(gmap), fr.new_images(with_counts=True))
    torch.cuda.synchronize()
    out = images_host(fr, img)[0]
    assert np.isfinite(out["rgb"]).all() and np.isfinite(out["depth"]).all()
    assert (out["last"] <= n).all() and (img["n_contrib"] <= n).all()


@pytest.mark.parametrize("capacity", [0, 1, 5, 12])
def test_items_beyond_the_ordered_capacity(capacity):
    """The grids are sized by the item order's capacity; a batch with more items (then not ordered)
    is still rendered and differentiated completely: 4 tiles of 8 items here."""
    gmap, _ = _stack(50, -1.0)
    cam = Camera(40.0, 40.0, 14.5, 13.0, 29, 26, np.eye(3, dtype=np.float32), np.zeros(3, np.float32))
    gm = gs.GaussianMapTensors.from_numpy(gmap)
    out = []
    for cut in (None, capacity):
        fr = gs.Frame(50, [cam])
        assert fr.n_items == 32
        if cut is not None:
            fr.c_bins.item_capacity = cut
        img = fr.forward(gm)
        g = fr.render_bwd(gm, img, torch.ones_like(img["rgb"]), torch.ones_like(img["depth"]))
        torch.cuda.synchronize()
        fr.check_status()
        out.append((img, g))
    for k in ("rgb", "depth", "unc", "T", "last"):
        assert torch.equal(out[0][0][k], out[1][0][k])
    for k in ("dmo", "dsu", "dq", "drgb"):      # (sums of atomics: equal up to their order)
        a, b = out[0][1][k], out[1][1][k]
        assert float((a - b).abs().max()) <= 1e-4 * float(a.abs().max())


@pytest.mark.parametrize("logit", [-6.5, -2.0])     # nothing saturates; everything does, early in the list
@pytest.mark.parametrize("n", [1023, 1025, 1120, 1153, 2500, 4099])
def test_long_lists_of_the_information_gain(n, logit):
    """Lists long enough to be shared by a block's warps (above 1,024 entries; rounds of 96): the
    score is the oracle's, and bit for bit that of the same pixels in other tiles and chunk depths."""
    gmap, cams = _stack(n, logit)
    gmap.mo[:, 2] = 2.0 + np.arange(n) * np.float32(0.002)
    gmap.mo[:, 3] = logit
    gm = gs.GaussianMapTensors.from_numpy(gmap)
    prm = gs.RenderParams(alpha_min=1e-3)
    ref = O.render_images(gmap, cams, O.Params(16, 16, prm.eps2d, prm.near, prm.guard, prm.alpha_min, prm.alpha_max,
                                               prm.T_min))[0]
    got = [float(gs.InfoGain(n, cams, gs.RenderParams(alpha_min=1e-3, ig_batch=b))(gm)[0]) for b in gs.IG_BATCH_CANDIDATES]
    assert got[0] == got[1] == got[2]
    # a skip or stop decision within rounding moves a pixel by at most alpha_min or T_min times u <= 1
    slack = ref["knife"].mean() * max(prm.alpha_min, prm.T_min)
    assert abs(got[0] - ref["unc"].mean()) <= IG_RTOL * abs(ref["unc"].mean()) + 1e-7 + slack


@pytest.mark.parametrize("capacity", [0, 1, 5, 100, 1023])
def test_items_beyond_the_ordered_capacity_of_large_images(capacity):
    """The same for more possible items than one wave of blocks has (128 tiles, 4,096 of 3,648),
    where a second launch looks for the items beyond the capacity."""
    gmap, _ = _stack(50, -1.0)
    cam = Camera(400.0, 400.0, 125.0, 60.0, 250, 120, np.eye(3, dtype=np.float32), np.zeros(3, np.float32))
    gm = gs.GaussianMapTensors.from_numpy(gmap)
    out = []
    for cut in (None, capacity):
        fr = gs.Frame(50, [cam])
        assert fr.n_items == 1024 and fr.n_tiles == 128
        if cut is not None:
            fr.c_bins.item_capacity = cut
        img = fr.forward(gm)
        g = fr.render_bwd(gm, img, torch.ones_like(img["rgb"]), torch.ones_like(img["depth"]))
        torch.cuda.synchronize()
        fr.check_status()
        out.append((img, g))
    for k in ("rgb", "depth", "unc", "T", "last"):
        assert torch.equal(out[0][0][k], out[1][0][k])
    for k in ("dmo", "dsu", "dq", "drgb"):      # (sums of atomics: equal up to their order)
        a, b = out[0][1][k], out[1][1][k]
        assert float((a - b).abs().max()) <= 1e-4 * float(a.abs().max())


def test_chunk_depth_one_is_depth_two():
    gmap, cams = _stack(33, 0.0)
    gm = gs.GaussianMapTensors.from_numpy(gmap)
    a, b = (gs.Frame(33, cams, gs.RenderParams(fwd_batch=k)).forward(gm) for k in (1, 2))
    for k in ("rgb", "depth", "unc", "T", "last"):
        assert torch.equal(a[k], b[k])


@pytest.mark.parametrize("n", [1, 2, 3, 5, 9, 33, 61])
def test_staged_leftovers_never_count_without_an_opacity_floor(n):
    """alpha_min = 0 again, with infinite colours and uncertainties staged beforehand in every slot of
    the rings (a longer stack): the forward with and without counts and the information gain at
    every chunk depth give the oracle's values."""
    gmap, cams = _stack(n, -1.0)
    long, _ = _stack(200, -6.0)          # transparent: its 200 entries all pass through the ring
    su = long.su.copy()
    su[:, 3] = np.inf
    hot = gs.GaussianMapTensors.from_numpy(GaussianMap(long.mo, su, long.q, np.full_like(long.rgb, np.inf)))
    gm = gs.GaussianMapTensors.from_numpy(gmap)
    P = O.Params(16, 16, 0.3, 0.2, 1.3, 0.0, 0.99, 1e-4)
    ref = O.render_images(gmap, cams, P)[0]
    ok = ~ref["knife"]
    for b in gs.FWD_BATCH_CANDIDATES:
        prm = gs.RenderParams(alpha_min=0.0, fwd_batch=b)
        for counts in (False, True):
            for _ in range(3):
                gs.Frame(200, cams, prm).forward(hot)
            fr = gs.Frame(n, cams, prm)
            h = images_host(fr, fr.forward(gm, fr.new_images(with_counts=counts)))[0]
            for k in ("rgb", "unc", "T"):
                np.testing.assert_allclose(h[k][ok], ref[k][ok], rtol=0, atol=IMG_ATOL, err_msg=k)
            np.testing.assert_allclose(h["depth"][ok], ref["depth"][ok], rtol=0, atol=DEPTH_RTOL * (2.0 + 0.01 * n))
            assert (h["last"] <= n).all()
    # a pixel of a knife-edge decision moves by at most T_min times u <= 1
    slack = ref["knife"].mean() * 1e-4
    for b in gs.IG_BATCH_CANDIDATES:
        prm = gs.RenderParams(alpha_min=0.0, ig_batch=b)
        for _ in range(3):
            gs.InfoGain(200, cams, prm)(hot)
        ig = float(gs.InfoGain(n, cams, prm)(gm)[0])
        assert abs(ig - ref["unc"].mean()) <= IG_RTOL * abs(ref["unc"].mean()) + 1e-7 + slack


@pytest.mark.parametrize("n", [1, 2, 3, 5, 31, 33, 50])
def test_last_and_gradients_without_an_opacity_floor(n):
    """alpha_min = 0: every entry of the list counts and the padding of a last chunk does not, so
    `last` is the one-launch render's (it indexes the tile's list) and the adjoint, which replays
    the list from it, gives the oracle's gradients."""
    gmap, cams = _stack(n, -2.0)
    gm = gs.GaussianMapTensors.from_numpy(gmap)
    ref = O.render_images(gmap, cams, O.Params(16, 16, 0.3, 0.2, 1.3, 0.0, 0.99, 1e-4))[0]
    rng = np.random.default_rng(n)
    d = rng.normal(size=(9, 13, 4))
    d[ref["knife"]] = 0.0
    gref = O.grad(gmap, cams, [d], O.Params(16, 16, 0.3, 0.2, 1.3, 0.0, 0.99, 1e-4))
    d_rgb = torch.from_numpy(np.ascontiguousarray(d[..., :3].transpose(2, 0, 1)).reshape(-1)).float().cuda()
    d_dep = torch.from_numpy(np.ascontiguousarray(d[..., 3]).reshape(-1)).float().cuda()
    for b in gs.FWD_BATCH_CANDIDATES:
        prm = gs.RenderParams(alpha_min=0.0, fwd_batch=b)
        fr = gs.Frame(n, cams, prm)
        img = fr.forward(gm, fr.new_images(with_counts=True))
        small, status = gs.render_small(gm, cams, prm)
        assert int(status) == 0 and torch.equal(img["last"], small["last"])
        np.testing.assert_array_equal(img["n_contrib"].cpu().numpy().reshape(9, 13)[~ref["knife"]],
                                      ref["n_contrib"][~ref["knife"]])
        out = fr.render_bwd(gm, img, d_rgb, d_dep)
        for k in ("dmo", "dsu", "dq", "drgb"):
            a, g = out[k].cpu().numpy().astype(np.float64), gref[k]
            np.testing.assert_allclose(a, g, rtol=0, atol=GRAD_RTOL * np.abs(g).max() + 1e-7, err_msg=k)
