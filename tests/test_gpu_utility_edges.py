"""Edges of the planner kernels' groups, chunks and windows against the oracle: groups of 32
Gaussians with a bounding sphere (view utility, collision), chunks of 2,048 Gaussians and
groups of 8 warps of points (collision), block sums in shared memory up to 2,048 regions,
maps whose neighbours lie together and maps in random order."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2409_18122_gb300 import gs, scenes

pytestmark = pytest.mark.gpu


def _map(n, order, seed=3):
    g = scenes.config3(seed=seed, n=max(n, 64), n_side=1).gmap
    if order == "random":
        g = g.subset(np.random.default_rng(seed).permutation(g.n))
    return g.subset(np.arange(n))


@pytest.mark.parametrize("order", ["patches", "random"])
@pytest.mark.parametrize("n,dims", [(1, (1, 1, 1)), (33, (4, 4, 2)), (5000, (16, 16, 8)), (5000, (683, 3, 1)),
                                    (70001, (4, 4, 2))])
def test_region_sums(n, dims, order):
    g = _map(n, order)
    size = 10.0 / dims[0]
    omega, count = gs.region_uncertainty(gs.GaussianMapTensors.from_numpy(g), (0.0, 0.0, 0.0), size, dims)
    ref, ref_cnt = O.region_uncertainty(g.mo, g.su[:, 3], (0.0, 0.0, 0.0), size, dims)
    np.testing.assert_array_equal(count.cpu().numpy(), ref_cnt)
    # FP64 sums rounded once to FP32
    np.testing.assert_allclose(omega.cpu().numpy(), ref, rtol=1e-6, atol=0)


@pytest.mark.parametrize("n", [1, 31, 33, 4097])
def test_thresholds_edges(n):
    g = _map(n, "random")
    vu = gs.ViewUtility([scenes.yaw_camera(5, 5, 1.5, 0.3, 80, 60, 65.6)])
    st = vu.thresholds(gs.GaussianMapTensors.from_numpy(g)).cpu().numpy()
    ref = O.uncertainty_thresholds(g.mo, g.su[:, 3])
    assert st[4] == ref[4]
    np.testing.assert_allclose(st[:4], ref[:4], rtol=1e-13, atol=1e-15)


@pytest.mark.parametrize("order", ["patches", "random"])
@pytest.mark.parametrize("n,views", [(1, 1), (33, 31), (3000, 33), (20011, 257)])
def test_view_counts(n, views, order):
    g = _map(n, order)
    if n > 100:   # a mean that is not a number keeps its group from being culled and is never visible
        g.mo[n // 2, 0] = np.nan
        g.mo[n // 3, 1] = np.inf
    rng = np.random.default_rng(views)
    cams = []
    for i in range(views):
        c = scenes.yaw_camera(*rng.uniform([0, 0, 0.5], [10, 10, 2.5]), rng.uniform(0, 6.28), 80 + i % 3, 60, 65.6)
        if i % 5 == 1:
            c.R = (c.R * np.float32(1.5)).astype(np.float32)   # not a rotation: the test is defined by its arithmetic
        if i % 5 == 2:
            c.cx, c.cy = -20.0, 200.0                          # principal point outside the image
        cams.append(c)
    gm = gs.GaussianMapTensors.from_numpy(g)
    vu = gs.ViewUtility(cams)
    st = vu.thresholds(gm).cpu().numpy()
    xi = vu(gm).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref_xi, ref_cnt = O.view_utility(g.mo, g.su[:, 3], cams, thresholds=tuple(float(x) for x in st))
    np.testing.assert_array_equal(vu.counts.cpu().numpy().astype(np.int64), ref_cnt)
    np.testing.assert_array_equal(xi, ref_xi.astype(np.float32))


@pytest.mark.parametrize("order", ["patches", "random"])
@pytest.mark.parametrize("n,points", [(1, 1), (32, 7), (33, 9), (2048, 129), (2049, 33), (20011, 300)])
def test_collision_edges(n, points, order):
    g = _map(n, order)
    if n > 100:
        g.mo[n // 2, 0] = np.nan
        g.mo[n // 3, 1] = np.inf
    rng = np.random.default_rng(n)
    pts = np.zeros((points, 4), np.float32)
    pts[:, :3] = rng.uniform([-1, -1, 0.0], [11, 11, 3], (points, 3))
    gm = gs.GaussianMapTensors.from_numpy(g)
    for r_robot, lam, gz in ((0.2, 3.0, float("-inf")), (0.0, 0.0, 0.5), (0.05, 1.0, 100.0)):
        margin, hit = gs.collision_check(gm, torch.from_numpy(pts).cuda(), r_robot, lam, gz)
        keep = np.isfinite(g.mo[:, :3]).all(1)      # others take part in nothing
        ref_m, ref_h = O.collision_check(g.mo[keep], g.su[keep], pts, r_robot, lam, gz)
        np.testing.assert_array_equal(hit.cpu().numpy().astype(bool), ref_h)
        # |p - mu| - gamma in FP32: a few units in the last place of |p - mu| and gamma
        np.testing.assert_allclose(margin.cpu().numpy(), ref_m, rtol=1e-5, atol=2e-6)


@pytest.mark.parametrize("points", [9, 33, 129, 257, 1000])
@pytest.mark.parametrize("order", ["random", "half"])
def test_collision_of_maps_in_random_order(order, points):
    """Maps whose neighbours in memory are not neighbours in space: most groups matter to most
    points, which then take whole chunks."""
    n = 40_003
    g = _map(n, "random" if order == "random" else "patches")
    if order == "half":      # chunks of both kinds
        p = np.arange(n)
        p[n // 2:] = np.random.default_rng(1).permutation(p[n // 2:])
        g = g.subset(p)
    g.mo[n // 2, 0], g.mo[n // 3, 1] = np.nan, np.inf
    rng = np.random.default_rng(points)
    pts = np.zeros((points, 4), np.float32)
    pts[:, :3] = rng.uniform([-1, -1, 0.0], [11, 11, 3], (points, 3))
    pts[0, :3] = g.mo[7, :3]
    gm = gs.GaussianMapTensors.from_numpy(g)
    for r_robot, lam, gz in ((0.2, 3.0, float("-inf")), (0.0, 0.0, 0.5)):
        margin, hit = gs.collision_check(gm, torch.from_numpy(pts).cuda(), r_robot, lam, gz)
        keep = np.isfinite(g.mo[:, :3]).all(1)
        ref_m, ref_h = O.collision_check(g.mo[keep], g.su[keep], pts, r_robot, lam, gz)
        np.testing.assert_array_equal(hit.cpu().numpy().astype(bool), ref_h)
        np.testing.assert_allclose(margin.cpu().numpy(), ref_m, rtol=1e-5, atol=2e-6)
        # what the other points are does not matter
        some = rng.choice(points, min(points, 9), replace=False)
        for i in some:
            m1, h1 = gs.collision_check(gm, torch.from_numpy(pts[i:i + 1]).cuda(), r_robot, lam, gz)
            assert float(m1[0]) == float(margin[i]) and int(h1[0]) == int(hit[i])


@pytest.mark.parametrize("regions", [7, 8, 9, 33])
def test_region_tables(regions):
    """A warp's table of eight regions: not full, exactly full, overflowing, and regions that come
    back after the table is full (in rounds of all regions, and then the first ones again)."""
    n = 64 * 40
    rng = np.random.default_rng(regions)
    g = _map(n, "random")
    r = np.arange(n) // 5 % regions
    r[n // 2:] = rng.integers(0, regions, n - n // 2)
    g.mo[:, 0] = r + rng.uniform(0.1, 0.9, n)
    g.mo[:, 1:3] = 0.5
    g.mo[::97, 0] = -1.0       # outside the grid
    omega, count = gs.region_uncertainty(gs.GaussianMapTensors.from_numpy(g), (0.0, 0.0, 0.0), 1.0, (regions, 1, 1))
    ref, ref_cnt = O.region_uncertainty(g.mo, g.su[:, 3], (0.0, 0.0, 0.0), 1.0, (regions, 1, 1))
    np.testing.assert_array_equal(count.cpu().numpy(), ref_cnt)
    np.testing.assert_allclose(omega.cpu().numpy(), ref, rtol=1e-6, atol=0)


@pytest.mark.parametrize("views", [1, 31, 100, 257])
@pytest.mark.parametrize("n", [1, 65, 19_456, 19_457, 38_913, 77_825, 155_648, 155_649])
def test_view_counts_of_maps_with_fewer_groups_than_warps(n, views):
    """Groups shared by eight, four and two warps, one each, and more than one per warp (4,864 warps
    on 152 multiprocessors), with view counts that do not divide; both modes."""
    g = _map(n, "random")
    rng = np.random.default_rng(n + views)
    cams = [scenes.yaw_camera(*rng.uniform([0, 0, 0.5], [10, 10, 2.5]), rng.uniform(0, 6.28), 80, 60, 65.6)
            for _ in range(views)]
    gm = gs.GaussianMapTensors.from_numpy(g)
    vu = gs.ViewUtility(cams)
    st = vu.thresholds(gm).cpu().numpy()
    vu(gm)
    ref_xi, ref_cnt = O.view_utility(g.mo, g.su[:, 3], cams, thresholds=tuple(float(x) for x in st))
    np.testing.assert_array_equal(vu.counts.cpu().numpy().astype(np.int64), ref_cnt)
    np.testing.assert_array_equal(vu.xi.cpu().numpy(), ref_xi.astype(np.float32))
    sums = vu(gm, 1).cpu().numpy()
    ref = O.view_utility(g.mo, g.su[:, 3], cams, mode="sum")[0]
    # positive terms through about 40 roundings to FP32 (5 + 2 per warp, 8 per block, 19 + 5 over blocks)
    np.testing.assert_allclose(sums, ref, rtol=3e-6, atol=0)
