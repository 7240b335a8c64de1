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
