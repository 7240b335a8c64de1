"""The record sort at its edges: record counts around its tiles (1,024 keys for capacities up to
2^20 records, 4,096 above), and keys whose top 14 bits span 511 (three passes) or 512 (four),
from an aligned and an unaligned smallest key.  Whole numbers: the oracle's lists exactly."""
import numpy as np
import pytest

from paper_2409_18122_gb300 import scenes
from paper_2409_18122_gb300.scenes import Camera

from test_gpu_parity import _bin_only, _check_bins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("top,base", [(511, 0x3E4CCCCD), (512, 0x3E4CCCCD), (511, 0x3E400000), (512, 0x3E43FFFF)])
@pytest.mark.parametrize("n", [1023, 1025, 4095, 4097, 8193])
def test_tile_and_span_edges(n, top, base, large):
    cams = [Camera(100, 100, 60, 40, 120, 80), Camera(50, 50, 8, 8, 17, 9), Camera(100, 100, 160, 120, 320, 240)]
    rec = scenes.synthetic_records(n + top, n, cams, max_extent=5, tie_frac=0.2)
    rng = np.random.default_rng(n)
    R = len(rec["gid"])
    lo = base >> 18
    dkey = ((lo + rng.integers(0, top + 1, R, dtype=np.uint64)) << 18 | rng.integers(0, 1 << 18, R, dtype=np.uint64))
    dkey = np.maximum(dkey, base).astype(np.uint32)
    dkey[: R // 4] = dkey[R // 4: 2 * (R // 4)]
    dkey[R // 3], dkey[R // 2] = base, (lo + top) << 18 | 5
    assert int(dkey.max() >> 18) - int(dkey.min() >> 18) == top and int(dkey.min()) == base
    rec["dkey"] = dkey
    if large:
        rec["gid"][-1] = 400_000      # a frame of 400,001 Gaussians and three views: the large tiles
    fr = _bin_only(rec, cams)
    assert (fr.rec_capacity > 1 << 20) == large
    _check_bins(fr, rec, cams)
    fr.check_status()


@pytest.mark.parametrize("views", [31, 32, 200])
@pytest.mark.parametrize("n_cap", [3000, 6144, 6145, 40_000])
def test_many_views(n_cap, views):
    """Many segments of few partitions (one scan block per view), of at most a tile and a half or
    more records (the two tile sizes), one view holding most of the records and some none."""
    cams = [Camera(40, 40, 20, 10, 40 + 3 * (i % 5), 20) for i in range(views)]
    rng = np.random.default_rng(n_cap + views)
    most = int(rng.integers(0, views))
    gid, view, rect = [], [], []
    for v, c in enumerate(cams):
        k = min(n_cap, 12_000) if v == most else int(rng.choice([0, 1, 33, 150]))
        gid.append(np.sort(rng.choice(n_cap, k, replace=False)).astype(np.uint32))
        view.append(np.full(k, v, np.uint32))
        tx, ty = -(-c.width // 16), -(-c.height // 16)
        x0, y0 = rng.integers(0, tx, k), rng.integers(0, ty, k)
        rect.append(np.stack([x0, y0, x0 + 1 + rng.integers(0, tx - x0), y0 + 1 + rng.integers(0, ty - y0)], 1))
    rec = dict(gid=np.concatenate(gid), view=np.concatenate(view), rect=np.concatenate(rect).astype(np.int32))
    rec["dkey"] = rng.uniform(0.2, 30.0, len(rec["gid"])).astype(np.float32).view(np.uint32)
    rec["dkey"][::3] = rec["dkey"][0]
    rec["gid"][-1] = n_cap - 1        # (the frame's Gaussians)
    fr = _bin_only(rec, cams)
    assert fr.rec_capacity == n_cap * views
    _check_bins(fr, rec, cams)
    fr.check_status()
