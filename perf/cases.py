"""Workloads of the splatting path, timed through the package's public entry points.

Each case is one pass of what a user's program repeats: a render, a mapping iteration up to
its gradients, a batch of scored candidate views, the render-free planner quantities, the
collision check of a trajectory, an optimiser update.  Inputs are synthetic, drawn on the GPU
from the seed alone, with the distributions of `paper_2409_18122_gb300.scenes`: a 10 x 10 m
room with 50 planar patches, a 40 x 40 m map with 750, or a box of uniform means.

`exact` computes the same outputs in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_2409_18122_gb300 import gs, scenes

DEV = "cuda"
NEAR, GUARD, EPS2D, AMIN, AMAX, TMIN = 0.2, 1.3, 0.3, 1.0 / 255.0, 0.99, 1e-4
MIX = "80x60,160x120,320x240"          # candidate resolutions of a planning step
MIX_TILES = "8x8,16x16,32x16"          # ... and the tiles the autotuner picks for them
L1, EQ3 = (0.1, 1.0 / 3.0, 0.0), (1.0, 0.4, 0.1)


def listed():
    return [
        # A 2,000-Gaussian preview in one launch: the smallest call, all latency.
        dict(name="small_2k", kind="small", n=2000, views=1, sizes="128x96", tiles="16x16"),
        # Tracking or display: one 640x480 view of a young map.
        dict(name="render_200k", kind="render", n=200000, views=1, sizes="640x480", tiles="16x16"),
        # Ragged views of an odd-sized map: images that end inside tiles, two tile shapes.
        dict(name="render_50k_ragged", kind="render", n=50021, views=3, sizes="333x217,97x131", tiles="16x16,8x8"),
        # The mapping iteration: 500k Gaussians, four 640x480 keyframes, L1 loss, adjoint.
        dict(name="train_500k", kind="train", n=500000, views=4, sizes="640x480", tiles="16x16", loss="l1",
             autograd=False),
        # The large map's mapping iteration with the full loss (SSIM): eight 1280x720 keyframes.
        dict(name="train_3m", kind="train", n=3000000, views=8, sizes="1280x720", tiles="32x32", loss="eq3",
             autograd=False),
        # A small map refined through autograd, odd image size: launches and host work count.
        dict(name="train_20k_autograd", kind="train", n=20011, views=2, sizes="321x243", tiles="16x16", loss="eq3",
             autograd=True),
        # The planning step: 256 candidate views at three resolutions over 1M Gaussians.
        dict(name="ig_1m_256", kind="ig", n=1000000, views=256, sizes=MIX, tiles=MIX_TILES),
        # A few candidates over a young map, default tiles.
        dict(name="ig_200k_27", kind="ig", n=200003, views=27, sizes=MIX, tiles="16x16"),
        # Candidates over the large map.
        dict(name="ig_3m_384", kind="ig", n=3000000, views=384, sizes="160x120,320x240", tiles="16x16,32x16"),
        # Render-free planning after a map update: uncertainties, thresholds, regions, xi.
        dict(name="plan_1m_256", kind="plan", n=1000000, views=256, sizes=MIX, states=0),
        # The test points of one trajectory against every Gaussian of the large map.
        dict(name="collision_3m_129", kind="collision", n=3000000, points=129),
        # The optimiser update of the 500k-Gaussian map.
        dict(name="adam_500k", kind="adam", n=500000),
    ]


def draw(rng):
    def logu(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def size(lo, hi):
        w = logu(lo, hi)
        return "%dx%d" % (w, max(17, int(w * rng.uniform(0.55, 0.8))))

    tile = lambda: rng.choice(["16x16", "16x8", "8x8", "32x8", "32x16", "32x32"])  # noqa: E731
    kind = rng.choice(["small", "render", "render", "train", "train", "ig", "ig", "plan", "collision", "adam"])
    if kind == "small":
        return dict(kind=kind, n=logu(150, 2000), views=rng.randint(1, 3), sizes=size(48, 160), tiles=tile())
    if kind == "render":
        return dict(kind=kind, n=logu(5000, 500000), views=rng.randint(1, 4), sizes=size(64, 800), tiles=tile())
    if kind == "train":
        return dict(kind=kind, n=logu(5000, 1000000), views=rng.randint(1, 4), sizes=size(64, 800), tiles=tile(),
                    loss=rng.choice(["l1", "eq3"]), autograd=rng.random() < 0.5)
    if kind == "ig":
        sizes = rng.choice([MIX, "160x120,320x240", "%s,%s" % (size(40, 330), size(40, 330))])
        return dict(kind=kind, n=logu(20000, 1000000), views=logu(4, 256), sizes=sizes,
                    tiles=",".join(tile() for _ in sizes.split(",")))
    if kind == "plan":
        states = rng.choice([0, 0, 4])
        views = logu(4, 512)
        return dict(kind=kind, n=logu(20000, 3000000), views=views - views % 4 if states else views, sizes=MIX,
                    states=states)
    if kind == "collision":
        return dict(kind=kind, n=logu(20000, 3000000), points=logu(16, 1000))
    return dict(kind=kind, n=logu(20000, 3000000))


# ------------------------------------------------------------------------------- inputs
def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + salt)


def _large(case):
    return case["n"] >= 2000000


def _map(case, seed):
    """(mo, su, q, rgb) float32 [n, 4]."""
    n, g = case["n"], _gen(seed, 1)
    r = lambda *s: torch.rand(*s, generator=g, device=DEV)  # noqa: E731
    z = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    if case["kind"] == "small":
        mu = r(n, 3) * 4.0 + torch.tensor([-2.0, -2.0, 1.0], device=DEV)
    else:
        ext, patches = (40.0, 750) if _large(case) else (10.0, 50)
        centre = r(patches, 3) * torch.tensor([ext, ext, 3.0], device=DEV)
        nrm = torch.nn.functional.normalize(z(patches, 3), dim=1)
        side = 0.5 + 1.5 * r(patches)
        axis = torch.tensor([1.0, 0.0, 0.0], device=DEV).expand(patches, 3)
        other = torch.tensor([0.0, 1.0, 0.0], device=DEV).expand(patches, 3)
        e1 = torch.nn.functional.normalize(torch.linalg.cross(nrm, torch.where(nrm[:, :1].abs() < 0.9, axis, other)),
                                           dim=1)
        e2 = torch.linalg.cross(nrm, e1)
        p = (torch.arange(n, device=DEV) * patches) // n      # a patch's Gaussians are neighbours in the map
        a, b = (r(n) - 0.5) * side[p], (r(n) - 0.5) * side[p]
        mu = centre[p] + a[:, None] * e1[p] + b[:, None] * e2[p] + (0.02 * z(n))[:, None] * nrm[p]
    mo = torch.cat([mu, z(n, 1)], 1)
    su = torch.cat([-3.0 + 0.5 * z(n, 3), r(n, 1)], 1)
    q = torch.nn.functional.normalize(z(n, 4), dim=1)
    rgb = torch.cat([r(n, 3), torch.zeros(n, 1, device=DEV)], 1)
    return [t.contiguous() for t in (mo, su, q, rgb)]


def _cams(case, seed):
    """Plain cameras: dicts of fx, fy, cx, cy, w, h, R (camera to world), T, tile."""
    rng = np.random.default_rng([int(seed), 2])
    sizes = [tuple(int(x) for x in s.split("x")) for s in case["sizes"].split(",")]
    tiles = [tuple(int(x) for x in s.split("x")) for s in case.get("tiles", "16x16").split(",")]
    ext = 40.0 if _large(case) else 10.0
    side = max(1, math.ceil(math.sqrt(case["views"])))
    at = np.linspace(0.5, ext - 0.5, side) if side > 1 else np.array([ext / 2])
    out = []
    for i in range(case["views"]):
        k = i % len(sizes)
        w, h = sizes[k]
        if case["kind"] == "small":          # at the origin, looking along +z
            R, T, f = np.eye(3), np.array([0.1 * i, 0.0, 0.0]), 100.0 / 128.0 * w
        else:
            if case["kind"] in ("ig", "plan"):       # candidate lattice, random heading
                x, y, zc, yaw = at[i % side], at[i // side], 1.5, rng.uniform(0.0, 2 * np.pi)
            else:                                    # keyframe: looks towards the middle of the room
                x, y = rng.uniform(0.5, ext - 0.5, size=2)
                zc = rng.uniform(1.0, 2.0)
                yaw = np.arctan2(ext / 2 - y, ext / 2 - x) + rng.uniform(-np.pi / 4, np.pi / 4)
            fwd, down = np.array([np.cos(yaw), np.sin(yaw), 0.0]), np.array([0.0, 0.0, -1.0])
            R, T, f = np.stack([np.cross(down, fwd), down, fwd], axis=1), np.array([x, y, zc]), 0.8203125 * w
        f32 = lambda v: np.asarray(v, np.float32)  # noqa: E731
        out.append(dict(f=float(f32(f)), cx=w / 2.0, cy=h / 2.0, w=w, h=h, R=f32(R), T=f32(T),
                        tile=tiles[k % len(tiles)]))
    return out


def _cameras(case, seed):
    return [scenes.Camera(c["f"], c["f"], c["cx"], c["cy"], c["w"], c["h"], c["R"], c["T"], *c["tile"])
            for c in _cams(case, seed)]


def _targets(case, seed):
    """Observed images (flat, the layout of the rendered ones): smooth fields plus noise."""
    g = _gen(seed, 3)
    rgb, dep = [], []
    for c in _cams(case, seed):
        y, x = torch.meshgrid(torch.arange(c["h"], device=DEV) / c["h"], torch.arange(c["w"], device=DEV) / c["w"],
                              indexing="ij")
        ph = 6.3 * torch.rand(4, generator=g, device=DEV)
        f = [0.5 + 0.2 * torch.sin(5.0 * x + 3.0 * y + ph[k]) for k in range(3)]
        im = torch.stack(f) + 0.05 * torch.randn(3, c["h"], c["w"], generator=g, device=DEV)
        rgb.append(im.clamp(0.0, 1.0).reshape(-1))
        dep.append((3.0 + torch.sin(4.0 * x + ph[3]) +
                    0.05 * torch.randn(c["h"], c["w"], generator=g, device=DEV)).reshape(-1))
    return torch.cat(rgb).float().contiguous(), torch.cat(dep).float().contiguous()


def _moved(case, seed, mo):
    """The means before the last mapping iterations: 70% of them have moved."""
    g = _gen(seed, 4)
    d = 0.05 * torch.randn(mo.shape[0], 3, generator=g, device=DEV)
    d *= (torch.rand(mo.shape[0], 1, generator=g, device=DEV) < 0.7).float()
    prev = mo.clone()
    prev[:, :3] += d
    return prev


def _points(case, seed):
    g = _gen(seed, 5)
    ext = 40.0 if _large(case) else 10.0
    p = torch.rand(case["points"], 4, generator=g, device=DEV) * torch.tensor([ext, ext, 2.3, 0.0], device=DEV)
    p[:, 2] += 0.2
    return p.contiguous()


def _adam_state(case, seed):
    """Parameters, gradients and moments of a map in the middle of its refinement (step 20)."""
    g = _gen(seed, 6)
    n = case["n"]
    p = [torch.randn(n, 4, generator=g, device=DEV) for _ in range(4)]
    grads = [1e-4 * torch.randn(n, 4, generator=g, device=DEV) for _ in range(4)]
    m = [1e-4 * torch.randn(n, 4, generator=g, device=DEV) for _ in range(4)]
    v = [1e-8 * torch.rand(n, 4, generator=g, device=DEV) + 1e-10 for _ in range(4)]
    return p, grads, m, v


REGIONS = {False: ((0.0, 0.0, -1.0), 2.5, (4, 4, 2)), True: ((0.0, 0.0, -1.0), 2.5, (16, 16, 2))}


def _sized(buffers, call):
    """Runs a first pass and gives the buffers the room that it asked for, as a program does once."""
    call()
    torch.cuda.synchronize()
    while buffers.grow_if_needed():
        call()
        torch.cuda.synchronize()
    return buffers


def prepare(case, seed):
    k = case["kind"]
    s = dict(kind=k)
    if k == "adam":
        p, grads, m, v = _adam_state(case, seed)
        for t, d in zip(p, grads):
            t.grad = d
        s["opt"] = gs.Adam(p, lr=1e-3)
        for dst, src in zip(s["opt"].m + s["opt"].v, m + v):
            dst.copy_(src)
        s["opt"].step_count.fill_(20)
        return s
    arrays = _map(case, seed)
    if k == "train" and case["autograd"]:
        s["leaves"] = [t.requires_grad_() for t in arrays]
    else:
        s["map"] = gs.GaussianMapTensors(*arrays)
    if k == "collision":
        s["points"] = _points(case, seed)
        return s
    cams = _cameras(case, seed)
    if k == "small":
        P = sum(c.width * c.height for c in cams)
        e = lambda n, t=torch.float32: torch.zeros(n, dtype=t, device=DEV)  # noqa: E731
        s["cams"] = gs.cameras_to_device(cams)
        s["images"] = dict(rgb=e(3 * P), depth=e(P), unc=e(P), T=e(P), last=e(P, torch.int32))
        s["status"] = e(1, torch.int32)
        tw, th = (int(x) for x in case["tiles"].split("x"))
        s["params"] = gs.RenderParams(tile_w=tw, tile_h=th)
    elif k == "render":
        s["frame"] = f = gs.Frame(case["n"], cams)
        _sized(f, lambda: f.forward(s["map"]))
    elif k == "train":
        s["frame"] = f = gs.Frame(case["n"], cams, with_pair_tiles=False)
        _sized(f, lambda: f.forward(gs.GaussianMapTensors(*arrays)))
        s["loss"] = gs.ImageLoss.for_cameras(cams, EQ3 if case["loss"] == "eq3" else L1)
        s["ref"] = _targets(case, seed)
        if not case["autograd"]:
            s["images"] = s["frame"].new_images()
            s["grads"] = {n: torch.empty(case["n"], 4, device=DEV) for n in ("dmo", "dsu", "dq", "drgb")}
    elif k == "ig":
        # the large map's records are bounded by what its views see; the room's by n * views
        cap = case["n"] * case["views"]
        s["ig"] = (gs.InfoGain(case["n"], cams, pair_capacity=cap // 2, record_capacity=cap // 3) if _large(case)
                   else gs.InfoGain(case["n"], cams))
        _sized(s["ig"], lambda: s["ig"](s["map"]))
    elif k == "plan":
        s["prev"] = _moved(case, seed, s["map"].mo)
        s["vu"] = gs.ViewUtility(cams)
        s["states"], s["regions"] = case["states"], REGIONS[_large(case)]
    return s


# --------------------------------------------------------------------------------- run
def run(s):
    k = s["kind"]
    if k == "small":
        return gs.render_small(s["map"], s["cams"], s["params"], images=s["images"], status=s["status"])[0]
    if k == "render":
        img = s["frame"].forward(s["map"])
        return {n: img[n] for n in ("rgb", "depth", "unc", "T", "last")}
    if k == "train" and "leaves" in s:
        for t in s["leaves"]:
            t.grad = None
        rgb, depth, unc = gs.render(*s["leaves"], s["frame"])
        loss = gs.image_loss(rgb, depth, *s["ref"], s["loss"])
        loss.backward()
        return [rgb.detach(), depth.detach(), unc, loss.detach()] + [t.grad for t in s["leaves"]]
    if k == "train":
        img = s["frame"].forward(s["map"], s["images"])
        loss, d_rgb, d_depth = s["loss"](img["rgb"], img["depth"], *s["ref"])
        g = s["frame"].render_bwd(s["map"], img, d_rgb, d_depth, s["grads"])
        return [img["rgb"], img["depth"], img["unc"], loss, d_rgb, d_depth] + [g[n] for n in ("dmo", "dsu", "dq", "drgb")]
    if k == "ig":
        return s["ig"](s["map"])
    if k == "plan":
        gs.uncertainty_update(s["prev"], s["map"].mo, s["map"].su)
        stats = s["vu"].thresholds(s["map"])
        omega, count = gs.region_uncertainty(s["map"], *s["regions"])
        if s["states"]:
            xi, best = gs.trajectory_utility(s["vu"], s["map"], s["vu"].V // s["states"], s["states"])
            return [s["map"].su, stats, omega, count, xi, best]
        return [s["map"].su, stats, omega, count, s["vu"](s["map"]), s["vu"].counts]
    if k == "collision":
        return gs.collision_check(s["map"], s["points"], 0.2)
    s["opt"].step()
    return [list(s["opt"].params), list(s["opt"].m), list(s["opt"].v)]


# -------------------------------------------------------------------------------- work
def work(case):
    """Bytes: the map and references read once, the results written once.  Operations: about 40
    per Gaussian and view (the frustum test and, for the fifth that is visible, the projection)
    and per pixel about 100 contributing Gaussians at 12 each (render and scoring) or 40 more
    (adjoint); two per tap of the separable SSIM windows; 11 per point and Gaussian."""
    k, n = case["kind"], case["n"]
    if k == "adam":
        return dict(bytes=4 * n * 4 * 7 * 4, flops=4 * n * 4 * 12)
    if k == "collision":
        return dict(bytes=32 * n + 24 * case["points"], flops=11 * n * case["points"])
    V = case["views"]
    sizes = [tuple(int(x) for x in s.split("x")) for s in case["sizes"].split(",")]
    P = sum(sizes[i % len(sizes)][0] * sizes[i % len(sizes)][1] for i in range(V))
    if k == "plan":
        return dict(bytes=n * (16 + 16 + 32), flops=n * (30 + 20 * V))
    flops = 40 * n * V + 1200 * P
    if k == "ig":
        return dict(bytes=48 * n + 4 * V, flops=flops)
    out = 4 * P * (3 + 1 + 1 + 1 + 1)
    if k != "train":
        return dict(bytes=64 * n + out, flops=flops)
    ssim = 3 * 8 * 2 * 11 * 2 if case["loss"] == "eq3" else 0
    return dict(bytes=64 * n + 64 * n + out + 2 * 16 * P, flops=flops + 4000 * P + (20 + ssim) * P + 300 * n)


# ------------------------------------------------------------------------ 64-bit values
def _project64(m, c):
    """Projection of all Gaussians into one view; differentiable.  m: the map's four arrays in
    64 bits.  Returns the visible ones' (depth order) mean, conic, opacity, depth, half-widths
    and indices."""
    mo, su, q, _ = m
    R = torch.tensor(c["R"], dtype=torch.float64, device=DEV)
    T = torch.tensor(c["T"], dtype=torch.float64, device=DEV)
    f = c["f"]
    with torch.no_grad():      # first what can be visible at all
        t = (mo[:, :3] - T) @ R
        tz = t[:, 2]
        ok = (tz > NEAR) & ~(t[:, 0].abs() > GUARD * 0.5 * c["w"] / f * tz) & \
            ~(t[:, 1].abs() > GUARD * 0.5 * c["h"] / f * tz) & (torch.sigmoid(mo[:, 3]) >= AMIN)
        idx = ok.nonzero().squeeze(1)
        idx = idx[torch.sort(tz[idx], stable=True)[1]]
    mo, su, q = mo[idx], su[idx], q[idx]
    t = (mo[:, :3] - T) @ R
    tx, ty, tz = t.unbind(1)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                      2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                      2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    A = Rq * torch.exp(su[:, None, :3])
    o0 = torch.zeros_like(tz)
    J = torch.stack([f / tz, o0, -f * tx / tz ** 2, o0, f / tz, -f * ty / tz ** 2], 1).view(-1, 2, 3)
    B = (J @ R.T) @ A
    S = B @ B.transpose(1, 2)
    a, b, d = S[:, 0, 0] + EPS2D, S[:, 0, 1], S[:, 1, 1] + EPS2D
    det = a * d - b * b
    op = torch.sigmoid(mo[:, 3])
    mean = torch.stack([f * tx / tz + c["cx"], f * ty / tz + c["cy"]], 1)
    conic = torch.stack([d / det, -b / det, a / det], 1)
    with torch.no_grad():
        Q = 2 * torch.log(op / AMIN)
        half = torch.stack([(Q * a).clamp_min(0).sqrt(), (Q * d).clamp_min(0).sqrt()], 1)
    return idx, mean, conic, op, tz, half


def _tile64(mean, conic, op, x0, y0, x1, y1):
    """Blend weights [L, pixels] and final transmittance of a tile's depth-ordered list."""
    y, x = torch.meshgrid(torch.arange(y0, y1, device=DEV, dtype=torch.float64) + 0.5,
                          torch.arange(x0, x1, device=DEV, dtype=torch.float64) + 0.5, indexing="ij")
    dx = mean[:, :1] - x.reshape(1, -1)
    dy = mean[:, 1:] - y.reshape(1, -1)
    q = conic[:, :1] * dx * dx + 2 * conic[:, 1:2] * dx * dy + conic[:, 2:] * dy * dy
    al = (op[:, None] * torch.exp(-0.5 * q)).clamp_max(AMAX)
    al = al * (al >= AMIN)
    s = torch.cumsum(torch.log1p(-al), 0)
    Ti = torch.exp(s)
    al = al * (Ti >= TMIN)
    # the stop rule: once T (1 - alpha) < T_min nothing more is added
    Tb = torch.cat([torch.ones_like(Ti[:1]), Ti[:-1]], 0)
    return al * Tb, torch.exp(torch.log1p(-al).sum(0))


def _tiles64(c, mean, half, tw=32, th=16):
    """(x0, y0, x1, y1, list) of every tile of a view that some Gaussian can reach."""
    lo, hi = torch.ceil(mean - 0.5 - half), torch.floor(mean - 0.5 + half)
    for y0 in range(0, c["h"], th):
        y1 = min(y0 + th, c["h"])
        row = ((lo[:, 1] < y1) & (hi[:, 1] >= y0) & (lo[:, 1] <= hi[:, 1]) & (lo[:, 0] <= hi[:, 0])).nonzero().squeeze(1)
        rl, rh = lo[row, 0], hi[row, 0]
        for x0 in range(0, c["w"], tw):
            x1 = min(x0 + tw, c["w"])
            li = row[(rl < x1) & (rh >= x0)]
            if li.numel():
                yield x0, y0, x1, y1, li


def _images64(m, cams):
    """Per view: [6, h, w] = rgb, depth, unc, T."""
    out = []
    with torch.no_grad():
        for c in cams:
            im = torch.zeros(6, c["h"], c["w"], dtype=torch.float64, device=DEV)
            im[5] = 1.0
            idx, mean, conic, op, tz, half = _project64(m, c)
            ch = torch.cat([m[3][idx, :3], tz[:, None], m[1][idx, 3:]], 1)
            for x0, y0, x1, y1, li in _tiles64(c, mean, half):
                w, T = _tile64(mean[li], conic[li], op[li], x0, y0, x1, y1)
                im[:5, y0:y1, x0:x1] = (ch[li].T @ w).view(5, y1 - y0, x1 - x0)
                im[5, y0:y1, x0:x1] = T.view(y1 - y0, x1 - x0)
            out.append(im)
    return out


def _grads64(m, cams, d_imgs):
    """Gradient with respect to the map's arrays of sum(d_img * (rgb, depth)) over the views."""
    leaves = [t.clone().requires_grad_() for t in m]
    for c, d in zip(cams, d_imgs):
        idx, mean, conic, op, tz, half = _project64(leaves, c)
        ch = torch.cat([leaves[3][idx, :3], tz[:, None]], 1)
        cut = [t.detach().requires_grad_() for t in (mean, conic, op, ch)]
        for x0, y0, x1, y1, li in _tiles64(c, mean.detach(), half):
            w, _ = _tile64(cut[0][li], cut[1][li], cut[2][li], x0, y0, x1, y1)
            (cut[3][li].T @ w).backward(d[:, y0:y1, x0:x1].reshape(4, -1))
        use = [(a, b.grad) for a, b in zip((mean, conic, op, ch), cut) if b.grad is not None]
        torch.autograd.backward([a for a, _ in use], [b for _, b in use])
    return [torch.zeros_like(t) if t.grad is None else t.grad for t in leaves]


def _flat(ims, rows):
    return torch.cat([im[rows].reshape(-1) for im in ims])


def _loss64(case, cams, ims, ref_rgb, ref_dep):
    """loss[4], and per view dL/d(rgb, depth) [4, h, w]."""
    wd, wc, ws = EQ3 if case["loss"] == "eq3" else L1
    P = sum(c["w"] * c["h"] for c in cams)
    k = torch.arange(11, dtype=torch.float64, device=DEV) - 5
    g = torch.exp(-k * k / (2 * 1.5 ** 2))
    g = g / g.sum()
    blur = lambda t: torch.nn.functional.conv2d(torch.nn.functional.conv2d(  # noqa: E731
        t[:, None], g.view(1, 1, 11, 1), padding=(5, 0)), g.view(1, 1, 1, 11), padding=(0, 5))[:, 0]
    l1d = l1c = ss = 0.0
    p = 0
    grads = []
    for c, im in zip(cams, ims):
        n = c["w"] * c["h"]
        y = ref_rgb[3 * p:3 * (p + n)].double().view(3, c["h"], c["w"])
        yd = ref_dep[p:p + n].double().view(c["h"], c["w"])
        p += n
        x = im[:4].clone().requires_grad_()
        d, col = (x[3] - yd).abs().sum(), (x[:3] - y).abs().sum()
        L = (wd * d + wc * col) / P
        if ws:
            mx, my = blur(x[:3]), blur(y)
            sx, sy, sxy = blur(x[:3] ** 2) - mx * mx, blur(y * y) - my * my, blur(x[:3] * y) - mx * my
            S = ((2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))).sum()
            L = L - ws * S / (3 * P)
            ss += float(S)
        L.backward()
        grads.append(x.grad)
        l1d, l1c = l1d + float(d), l1c + float(col)
    l1d, l1c, ss = l1d / P, l1c / P, ss / (3 * P) if ws else math.nan
    L = wd * l1d + wc * l1c + (ws * (1 - ss) if ws else 0.0)
    return torch.tensor([L, l1d, l1c, ss], dtype=torch.float64, device=DEV), grads


def _see64(mo, su, c, hi, lo):
    R = torch.tensor(c["R"], dtype=torch.float64, device=DEV)
    t = (mo[:, :3] - torch.tensor(c["T"], dtype=torch.float64, device=DEV)) @ R
    px, py = c["f"] * t[:, 0] / t[:, 2] + c["cx"], c["f"] * t[:, 1] / t[:, 2] + c["cy"]
    vis = (t[:, 2] > NEAR) & (t[:, 2] <= 5.0) & (px >= 0) & (px < c["w"]) & (py >= 0) & (py < c["h"])
    return (vis & hi).sum() - (vis & lo).sum()


def exact(case, seed):
    k = case["kind"]
    if k == "adam":
        p, grads, m, v = [[t.double() for t in ts] for ts in _adam_state(case, seed)]
        m = [0.9 * a + 0.1 * g for a, g in zip(m, grads)]
        v = [0.999 * a + 0.001 * g * g for a, g in zip(v, grads)]
        p = [a - 1e-3 / (1 - 0.9 ** 21) * b / ((c / (1 - 0.999 ** 21)).sqrt() + 1e-8) for a, b, c in zip(p, m, v)]
        return [p, m, v]
    m = [t.double() for t in _map(case, seed)]
    if k == "collision":
        pts = _points(case, seed).double()
        gamma = 0.2 + 3.0 * torch.exp(m[1][:, :3].max(1)[0])
        best = [((m[0][:, :3] - p[:3]).norm(dim=1) - gamma).min() for p in pts]
        return [torch.stack(best), None]        # the flags are decisions in 32 bits
    cams = _cams(case, seed)
    if k == "plan":
        mo = _map(case, seed)[0]
        d = (mo.double() - _moved(case, seed, mo).double())[:, :3].norm(dim=1)
        su = m[1].clone()
        su[:, 3] = torch.where(d > 0, d, su[:, 3])
        u = su[:, 3]
        mean, sig = u.mean(), u.std(unbiased=False)
        stats = torch.stack([mean, sig, mean + sig / 2, mean - sig / 2, torch.tensor(float(len(u)), device=DEV,
                                                                                     dtype=torch.float64)])
        (ox, oy, oz), size, dims = REGIONS[_large(case)]
        i = torch.floor((m[0][:, :3] - torch.tensor([ox, oy, oz], device=DEV, dtype=torch.float64)) / size).long()
        inside = ((i >= 0) & (i < torch.tensor(dims, device=DEV))).all(1)
        r = ((i[:, 2] * dims[1] + i[:, 1]) * dims[0] + i[:, 0])[inside]
        R = dims[0] * dims[1] * dims[2]
        tot = torch.zeros(R, dtype=torch.float64, device=DEV).index_add_(0, r, u[inside])
        cnt = torch.bincount(r, minlength=R)
        omega = torch.where(cnt > 0, tot / cnt.clamp_min(1), torch.zeros_like(tot))
        # u is rounded to 32 bits before it is classified
        xi = torch.stack([_see64(m[0], su, c, u.float().double() > stats[2], u.float().double() < stats[3])
                          for c in cams]).double()
        if case["states"]:
            return [su, stats, omega, None, xi.view(-1, case["states"]).sum(1), None]
        return [su, stats, omega, None, xi, None]
    pixels = sum(c["w"] * c["h"] for c in cams)
    if pixels > 1300000 or case["n"] > 500000 or len(cams) * case["n"] > 6000000:
        return None                              # too long in 64 bits
    ims = _images64(m, cams)
    rgb, dep, unc, T = (_flat(ims, r) for r in (slice(0, 3), 3, 4, 5))
    if k == "ig":
        return torch.stack([im[4].mean() for im in ims])
    if k in ("small", "render"):
        return dict(rgb=rgb, depth=dep, unc=unc, T=T, last=None)
    loss, d = _loss64(case, cams, ims, *_targets(case, seed))
    g = _grads64(m, cams, d)
    g[1][:, 3] = 0.0
    if case["autograd"]:
        return [rgb, dep, unc, loss[0]] + g
    return [rgb, dep, unc, loss, _flat(d, slice(0, 3)), _flat(d, 3)] + g
