"""Workloads of the depth-map library for timing: whole depth maps, the steps
around them and the proposal network, each through the binding a program
calls (paper_2104_06165_gb300.mvs), over the sizes and options of the
library's configurations.

Scenes are seeded: one textured background plane, four textured tilted quads
with blank patches, rendered on the GPU by ray casting, seen by a reference
camera and sources at viewing angles of 15 to 40 degrees.
"""
import math

import numpy as np
import torch

from paper_2104_06165_gb300 import mvs, proposals

DEV = "cuda"
D_LO, D_HI = 2.0, 8.0
Z_C = 5.0                      # depth of the point every camera looks at
N_SINUSOIDS = 24
# (radius, samples per axis): 11 x 11 at dilation 2 by 6 x 6 samples, the
# paper's default 5/7, 21 x 21 at dilation 2, the paper's dense windows
WINDOWS = ((5.0, 6), (7.0, 11), (10.0, 11), (6.0, 13), (8.0, 17))


def listed():
    return [
        # a preview or a tracking frame: the smallest map, where launches and
        # the last wave count (the small configuration: 6 x 6 samples, 4 sources)
        {"name": "depth_320x240", "kind": "depth", "W": 320, "H": 240, "n_src": 4, "radius": 5.0, "samples": 6,
         "iters": 3, "mixed": False, "n_prop": 0},
        # the paper's own window and source count on an image of odd size
        {"name": "depth_1511x1007", "kind": "depth", "W": 1511, "H": 1007, "n_src": 8, "radius": 7.0, "samples": 11,
         "iters": 8, "mixed": False, "n_prop": 0},
        # the full-resolution map: one photograph of a high-resolution set
        {"name": "depth_3072x2048", "kind": "depth", "W": 3072, "H": 2048, "n_src": 10, "radius": 10.0, "samples": 11,
         "iters": 8, "mixed": False, "n_prop": 0},
        # the second half of a learned run: iterations with four proposed
        # planes per pixel on a given state, mixed precision
        {"name": "depth_1536x1024_learned", "kind": "depth", "W": 1536, "H": 1024, "n_src": 10, "radius": 10.0,
         "samples": 11, "iters": 1, "mixed": True, "n_prop": 4},
        # all views of a small scene at uneven resolutions in one call
        {"name": "batch_6_views", "kind": "batch", "W": 1536, "H": 1024, "n_views": 6, "radius": 10.0, "samples": 11,
         "iters": 4},
        # scoring a given plane map with a dense window (the window study's 8/8)
        {"name": "plane_cost_1024x683", "kind": "plane_cost", "W": 1024, "H": 683, "n_src": 8, "radius": 8.0,
         "samples": 17, "mixed": False},
        # filling the unrecovered pixels of a full-resolution map (line fits,
        # their costs, the 4-label MRF, normals)
        {"name": "plane_infer_3072x2048", "kind": "plane_infer", "W": 3072, "H": 2048, "n_src": 10, "radius": 10.0,
         "samples": 11, "min_cost": False},
        # cross-view consistency of a full-resolution map against ten others
        {"name": "geo_filter_3072x2048", "kind": "geo_filter", "W": 3072, "H": 2048, "n_src": 10},
        # merging the filtered maps of a scene into one cloud
        {"name": "fuse_8_views", "kind": "fuse", "W": 2048, "H": 1365, "n_views": 8},
        # depth ranges of a full-resolution view from structure-from-motion points
        {"name": "sparse_range_3072x2048", "kind": "sparse_range", "W": 3072, "H": 2048, "n_src": 10, "points": 20000},
        # the proposal network on one view (forward pass and decoding)
        {"name": "propose_1536x1024", "kind": "propose", "W": 1536, "H": 1024},
        # one training example: forward, loss, backward, gradients out
        {"name": "train_512x384", "kind": "train", "W": 512, "H": 384},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("depth", "depth", "depth", "batch", "plane_cost", "plane_infer", "geo_filter", "fuse",
                       "sparse_range", "propose", "train"))
    W = int(_log_uniform(rng, 160, 3072))
    H = max(96, int(W * rng.uniform(0.6, 0.8)))
    if H > 2048:
        H = 2048
    c = {"kind": kind, "W": W, "H": H}
    if kind in ("depth", "plane_cost", "plane_infer"):
        c["radius"], c["samples"] = rng.choice(WINDOWS)
        c["n_src"] = rng.randint(3, 10)
    if kind == "depth":
        c["mixed"] = rng.random() < 0.3
        c["n_prop"] = rng.choice((0, 0, 0, 4))
        c["iters"] = rng.randint(1, 8)
        # no more work than the largest listed map (a window costs its samples
        # and something of its own)
        cost = W * H * c["n_src"] * (c["samples"] ** 2 + 60)
        c["iters"] = max(1, min(c["iters"], int(0.8 * 3072 * 2048 * 10 * 181 * 8 / cost)))
    elif kind == "batch":
        c["W"] = int(_log_uniform(rng, 160, 1536))
        c["H"] = max(96, int(c["W"] * rng.uniform(0.6, 0.67)))
        c["n_views"] = rng.randint(4, 6)
        c["radius"], c["samples"] = rng.choice(WINDOWS[:3])
        c["iters"] = rng.randint(1, 4)
    elif kind == "plane_cost":
        c["W"] = int(_log_uniform(rng, 160, 1536))
        c["H"] = max(96, int(c["W"] * rng.uniform(0.6, 0.67)))
        c["mixed"] = rng.random() < 0.3
    elif kind == "plane_infer":
        c["min_cost"] = rng.random() < 0.3
    elif kind == "geo_filter":
        c["n_src"] = rng.randint(3, 10)
    elif kind == "fuse":
        c["W"] = int(_log_uniform(rng, 160, 2048))
        c["H"] = max(96, int(c["W"] * rng.uniform(0.6, 0.67)))
        c["n_views"] = rng.randint(4, 8)
    elif kind == "sparse_range":
        c["n_src"] = rng.randint(3, 10)
        c["points"] = int(_log_uniform(rng, 1000, 20000))
    elif kind == "propose":
        c["W"], c["H"] = 16 * rng.randint(4, 96), 16 * rng.randint(4, 64)
    elif kind == "train":
        c["W"], c["H"] = 16 * rng.randint(4, 32), 16 * rng.randint(4, 24)
    return c


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
def _look_at(C):
    """World-to-camera rotation and translation of a camera at C that looks
    at (0, 0, Z_C)."""
    z = np.array([0.0, 0.0, Z_C]) - C
    z /= np.linalg.norm(z)
    x = np.cross([0.0, 1.0, 0.0], z)
    x /= np.linalg.norm(x)
    R = np.stack([x, np.cross(z, x), z])
    return R, -R @ C


class _Scene:
    """Planes and cameras of one seed; views are rendered on demand."""

    def __init__(self, seed, sizes, spread):
        rng = np.random.default_rng(seed)
        self.sizes = sizes
        self.cams = []
        n = len(sizes) - 1
        for v, (W, H) in enumerate(sizes):
            f = 300.0 * W / 320.0
            K = np.array([[f, 0.0, (W - 1) / 2.0], [0.0, f, (H - 1) / 2.0], [0.0, 0.0, 1.0]])
            if v == 0:
                R, t = np.eye(3), np.zeros(3)
            else:
                a = math.radians(spread[0] + (spread[1] - spread[0]) * (v - 1) / max(n - 1, 1))
                b = 2.0 * math.pi * v / n + rng.uniform(-0.2, 0.2)
                R, t = _look_at(np.array([0.0, 0.0, Z_C]) + Z_C * np.array(
                    [math.sin(a) * math.cos(b), math.sin(a) * math.sin(b), -math.cos(a)]))
            self.cams.append((K, R, t))
        f0 = 300.0 * sizes[0][0] / 320.0
        self.planes = []
        for q in range(5):
            tilt, az = math.radians(rng.uniform(0, 15 if q == 0 else 50)), rng.uniform(0, 2 * math.pi)
            nrm = np.array([math.sin(tilt) * math.cos(az), math.sin(tilt) * math.sin(az), -math.cos(tilt)])
            e1 = np.cross(nrm, [1.0, 0.0, 0.0])
            e1 /= np.linalg.norm(e1)
            e2 = np.cross(nrm, e1)
            if q == 0:      # the background
                centre, half = np.array([0.0, 0.0, 7.0]), 40.0
            else:           # one quad per image quadrant
                depth = rng.uniform(3.0, 5.8)
                u = (0.3 if q % 2 else 0.7) + rng.uniform(-0.08, 0.08)
                v = (0.3 if q < 3 else 0.7) + rng.uniform(-0.08, 0.08)
                W, H = sizes[0]
                centre = depth * np.array([(u - 0.5) * W / f0, (v - 0.5) * H / f0, 1.0])
                half = rng.uniform(0.15, 0.22) * W * depth / f0
            z = centre[2]
            lam = np.exp(rng.uniform(math.log(4.0), math.log(32.0), N_SINUSOIDS)) * z / f0
            ang = rng.uniform(0, math.pi, N_SINUSOIDS)
            amp = rng.uniform(0.5, 1.0, N_SINUSOIDS)
            amp *= 38.0 / math.sqrt(0.5 * np.sum(amp ** 2))
            self.planes.append({"n": nrm, "c": centre, "e1": e1, "e2": e2, "half": half, "blank": 0.7 * half if q else 0.0,
                                "grey": rng.uniform(70, 190), "freq": 2 * math.pi * np.stack(
                                    [np.cos(ang), np.sin(ang)]) / lam, "phase": rng.uniform(0, 2 * math.pi, N_SINUSOIDS),
                                "amp": amp})

    def view(self, v, image=True):
        """(uint8 image or None, plane map (H, W, 4) of the visible surface,
        textured mask) of view v, on the GPU."""
        W, H = self.sizes[v]
        K, R, t = self.cams[v]
        ten = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device=DEV)  # noqa: E731
        yy, xx = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float32),
                                torch.arange(W, device=DEV, dtype=torch.float32), indexing="ij")
        f = K[0, 0]
        ray = torch.stack([(xx - K[0, 2]) / f, (yy - K[1, 2]) / f, torch.ones_like(xx)], -1)
        dirs = (ray.reshape(-1, 3) @ ten(R)).reshape(H, W, 3)
        C = -R.T @ t
        best = torch.full((H, W), math.inf, device=DEV)
        which = torch.zeros((H, W), dtype=torch.int8, device=DEV)
        for q, p in enumerate(self.planes):
            lam = float((p["c"] - C) @ p["n"]) / (dirs @ ten(p["n"]))
            s1 = lam * (dirs @ ten(p["e1"])) + float((C - p["c"]) @ p["e1"])
            s2 = lam * (dirs @ ten(p["e2"])) + float((C - p["c"]) @ p["e2"])
            hit = (lam > 0) & (lam < best) & (s1.abs() <= p["half"]) & (s2.abs() <= p["half"])
            best = torch.where(hit, lam, best)
            which = torch.where(hit, torch.tensor(q, dtype=torch.int8, device=DEV), which)
        best = torch.where(torch.isfinite(best), best, torch.tensor(7.0, device=DEV))
        textured = torch.ones((H, W), dtype=torch.bool, device=DEV)
        grey = torch.full((H * W,), 128.0, device=DEV) if image else None
        plane = torch.empty((H, W, 4), device=DEV)
        plane[..., 3] = best      # rays have unit z in the camera frame
        for q, p in enumerate(self.planes):
            nc = ten(R @ p["n"])
            sel = (which == q)
            flip = torch.where((ray @ nc) > 0, -1.0, 1.0)
            plane[..., :3] = torch.where(sel[..., None], flip[..., None] * nc, plane[..., :3])
            at = sel.reshape(-1).nonzero()[:, 0]
            if not at.numel():
                continue
            for part in at.split(1 << 20):
                P = dirs.reshape(-1, 3)[part] * best.reshape(-1)[part][:, None]
                s = torch.stack([P @ ten(p["e1"]) + float((C - p["c"]) @ p["e1"]),
                                 P @ ten(p["e2"]) + float((C - p["c"]) @ p["e2"])], 1)
                blank = (s[:, 0].abs() <= p["blank"]) & (s[:, 1].abs() <= p["blank"])
                textured.view(-1)[part] = ~blank
                if image:
                    g = 128.0 + torch.sin(s @ ten(p["freq"]) + ten(p["phase"])) @ ten(p["amp"])
                    grey[part] = torch.where(blank, torch.tensor(p["grey"], device=DEV, dtype=torch.float32), g)
        img = grey.clamp(20.0, 235.0).round().to(torch.uint8).reshape(H, W) if image else None
        return img, plane, textured


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _random_planes(shape, g):
    """Random normals turned to the camera and depths over the whole range."""
    n = torch.randn(shape + (3,), generator=g, device=DEV)
    n[..., 2] = -n[..., 2].abs() - 0.5
    n /= n.norm(dim=-1, keepdim=True)
    d = D_LO + (D_HI - D_LO) * torch.rand(shape, generator=g, device=DEV)
    return torch.cat([n, d[..., None]], -1)


def _estimated(plane, textured, g, wrong=0.05, noise=3e-4):
    """A depth map as the iterations leave it: the surface to within noise
    where there is texture, random planes elsewhere and on a few pixels, and
    its costs."""
    H, W = textured.shape
    good = textured & (torch.rand((H, W), generator=g, device=DEV) >= wrong)
    near = plane.clone()
    near[..., 3] *= 1.0 + noise * torch.randn((H, W), generator=g, device=DEV)
    est = torch.where(good[..., None], near, _random_planes((H, W), g)).contiguous()
    cost = torch.where(good, 0.02 + 0.2 * torch.rand((H, W), generator=g, device=DEV), torch.tensor(2.0, device=DEV))
    return est, cost, good


def _context(sc, images):
    K, R, t = (np.stack(a) for a in zip(*sc.cams))
    return mvs.Context(K, R, t, images, stream=torch.cuda.current_stream())


def _noise_images(sc, g):
    """Images for the steps that read the geometry only."""
    return [torch.randint(20, 236, (H, W), generator=g, device=DEV, dtype=torch.uint8).cpu().numpy()
            for W, H in sc.sizes]


def _params(case, seed, **kw):
    return mvs.PMParams(win_radius=case["radius"], win_samples=case["samples"], d_lo=D_LO, d_hi=D_HI, seed=seed,
                        precision=1 if case.get("mixed") else 0, **kw)


def _view_sizes(case):
    """Full, two-thirds and half resolution in turn (uneven view sizes)."""
    W, H = case["W"], case["H"]
    return [(W, H) if v % 3 == 0 else (2 * W // 3, 2 * H // 3) if v % 3 == 1 else (W // 2, H // 2)
            for v in range(case["n_views"])]


def _net_inputs(sc, g):
    img, plane, textured = sc.view(0)
    est, cost, good = _estimated(plane, textured, g)
    return img.contiguous(), est, cost, plane.contiguous(), good.to(torch.uint8)


def prepare(case, seed):
    g = _generator(seed)
    W, H, kind = case["W"], case["H"], case["kind"]
    s = {"kind": kind}
    if kind in ("batch", "fuse"):
        sc = _Scene(seed, _view_sizes(case), (15.0, 40.0))
    elif kind in ("propose", "train"):
        sc = _Scene(seed, [(W, H)], (15.0, 40.0))
    else:
        sc = _Scene(seed, [(W, H)] * (1 + case["n_src"]), (15.0, 40.0))
        s["srcs"] = list(range(1, 1 + case["n_src"]))
    if kind in ("depth", "batch", "plane_cost", "plane_infer"):
        views = [sc.view(v) for v in range(len(sc.sizes))]
        s["ctx"] = _context(sc, [v[0].cpu().numpy() for v in views])
    elif kind in ("geo_filter", "fuse", "sparse_range"):
        views = [sc.view(v, image=False) for v in range(len(sc.sizes))]
        s["ctx"] = _context(sc, _noise_images(sc, g))

    if kind == "depth":
        s["plane"] = torch.empty((H, W, 4), device=DEV)
        s["cost"] = torch.empty((H, W), device=DEV)
        if case["n_prop"]:
            # the state after an iteration: half the textured pixels have found
            # their plane; proposals near the surface and away from it
            est, _, _ = _estimated(views[0][1], views[0][2], g, wrong=0.5)
            s["start"] = (est, torch.empty((H, W), device=DEV))
            mvs.mvs_plane_cost(s["ctx"].h, 0, s["srcs"], _params(case, seed), *s["start"])
            props = [_estimated(views[0][1], views[0][2], g, wrong=w, noise=3e-3)[0] for w in (0.2, 0.5, 0.8, 1.0)]
            s["proposals"] = torch.stack(props[:case["n_prop"]], 2).contiguous()
            s["params"] = _params(case, seed, iters=1 + case["iters"], phase_begin=2, init_mode=mvs.MVS_INIT_GIVEN,
                                  n_prop=case["n_prop"], proposals=s["proposals"])
        else:
            s["params"] = _params(case, seed, iters=case["iters"])
    elif kind == "batch":
        n = case["n_views"]
        s["refs"] = list(range(n))
        s["srcs"] = [[u for u in range(n) if u != v] for v in range(n)]
        s["params"] = _params(case, seed, iters=case["iters"])
        s["planes"] = [torch.empty((h, w, 4), device=DEV) for w, h in sc.sizes]
        s["costs"] = [torch.empty((h, w), device=DEV) for w, h in sc.sizes]
    elif kind == "plane_cost":
        s["params"] = _params(case, seed)
        s["plane"] = _estimated(views[0][1], views[0][2], g, wrong=0.3)[0]
        s["cost"] = torch.empty((H, W), device=DEV)
        s["view_cost"] = torch.empty((H, W, case["n_src"]), device=DEV)
    elif kind == "plane_infer":
        s["params"] = _params(case, seed)
        s["phi"] = mvs.PhiParams(selection=mvs.MVS_PHI_SELECT_MIN_COST if case["min_cost"] else mvs.MVS_PHI_SELECT_MRF)
        s["plane"], s["cost"], _ = _estimated(views[0][1], views[0][2], g)
    elif kind == "geo_filter":
        for v, (_, plane, textured) in enumerate(views):
            mvs.mvs_set_depth_map(s["ctx"].h, v, *_estimated(plane, textured, g)[:2])
        s["params"] = mvs.FilterParams()
        s["keep"] = torch.empty((H, W), dtype=torch.uint8, device=DEV)
        s["count"] = torch.empty((H, W), dtype=torch.int32, device=DEV)
    elif kind == "fuse":
        s["keep"] = []
        for v, (_, plane, textured) in enumerate(views):
            est, cost, good = _estimated(plane, textured, g)
            mvs.mvs_set_depth_map(s["ctx"].h, v, est, cost)
            s["keep"].append(good.to(torch.uint8))
        total = sum(w * h for w, h in sc.sizes)
        s["views"] = list(range(len(views)))
        s["points"] = torch.zeros((total, 4), device=DEV)
        s["src"] = torch.zeros((total, 2), dtype=torch.int32, device=DEV)
    elif kind == "sparse_range":
        s.update(_sparse(sc, views, case["points"], g))
        s["range"] = torch.empty((H, W, 2), device=DEV)
    else:
        s["inputs"] = _net_inputs(sc, g)
        s["net"] = _Net(W, H)
        if kind == "propose":
            s["Kinv"] = np.linalg.inv(sc.cams[0][0])
            s["proposals"] = torch.empty((H, W, proposals.K_PROP, 4), device=DEV)
    torch.cuda.synchronize()
    return s


class _Net:
    """Owns a proposal network with the trained weights."""

    def __init__(self, W, H):
        self.h = mvs.mvs_cnn_create(W, H, D_LO, D_HI, 0, torch.cuda.current_stream())
        proposals.load_weights(self.h)

    def __del__(self):
        mvs.mvs_cnn_destroy(self.h)


def _sparse(sc, views, n, g):
    """Structure-from-motion output: surface points seen through random
    pixels, visible where they project inside an image (one in ten missed),
    half a pixel of observation noise, a few wrong points."""
    n_views = len(views)
    X = torch.empty((n, 3), dtype=torch.float64, device=DEV)
    of = torch.randint(0, n_views, (n,), generator=g, device=DEV)
    place = torch.rand((n, 2), generator=g, device=DEV)
    cams = [[torch.as_tensor(a, dtype=torch.float64, device=DEV) for a in c] for c in sc.cams]
    for v, (K, R, t) in enumerate(cams):
        W, H = sc.sizes[v]
        at = (of == v).nonzero()[:, 0]
        u, w = (place[at, 0] * (W - 1)).round().long(), (place[at, 1] * (H - 1)).round().long()
        pix = torch.stack([u.double(), w.double(), torch.ones_like(u).double()], 1)
        d = views[v][1][w, u, 3].double()
        Kinv = torch.as_tensor(np.linalg.inv(sc.cams[v][0]), device=DEV)
        X[at] = (d[:, None] * (pix @ Kinv.T) - t) @ R
    vis = torch.zeros(n, dtype=torch.int64, device=DEV)
    obs = torch.full((n, 2), math.nan, dtype=torch.float64, device=DEV)
    for v, (K, R, t) in enumerate(cams):
        W, H = sc.sizes[v]
        q = (X @ R.T + t) @ K.T
        u, w = q[:, 0] / q[:, 2], q[:, 1] / q[:, 2]
        seen = (q[:, 2] > 0) & (u >= 0) & (u <= W - 1) & (w >= 0) & (w <= H - 1)
        seen &= torch.rand(n, generator=g, device=DEV) > 0.1
        vis |= seen.long() << v
        if v == 0:
            noisy = torch.stack([u, w], 1) + 0.5 * torch.randn((n, 2), generator=g, device=DEV)
            obs = torch.where(seen[:, None], noisy, obs)
    wrong = torch.rand(n, generator=g, device=DEV) < 0.02
    X = torch.where(wrong[:, None], X * (1.0 + 0.1 * torch.rand((n, 1), generator=g, device=DEV)), X)
    err = 0.5 * torch.randn((n, 2), generator=g, device=DEV).norm(dim=1).double()
    return {"X": X.contiguous(), "vis": vis, "obs": obs.contiguous(),
            "reproj": torch.where(wrong, err + 5.0, err).contiguous()}


def run(s):
    kind = s["kind"]
    if kind == "depth":
        if "start" in s:     # the map is refined in place
            s["plane"].copy_(s["start"][0])
            s["cost"].copy_(s["start"][1])
        mvs.mvs_patchmatch(s["ctx"].h, 0, s["srcs"], s["params"], s["plane"], s["cost"])
        return s["plane"], s["cost"]
    if kind == "batch":
        mvs.mvs_patchmatch_batch(s["ctx"].h, s["refs"], s["srcs"], s["params"], s["planes"], s["costs"])
        return s["planes"], s["costs"]
    if kind == "plane_cost":
        mvs.mvs_plane_cost(s["ctx"].h, 0, s["srcs"], s["params"], s["plane"], s["cost"], s["view_cost"])
        return s["cost"], s["view_cost"]
    if kind == "plane_infer":
        # the pixels of low cost stay, so the filled map can be filled again
        mvs.mvs_plane_infer(s["ctx"].h, 0, s["srcs"], s["params"], s["phi"], None, s["plane"], s["cost"])
        return s["plane"]
    if kind == "geo_filter":
        mvs.mvs_geo_filter(s["ctx"].h, 0, s["srcs"], s["params"], s["keep"], s["count"])
        return s["keep"], s["count"]
    if kind == "fuse":
        n = mvs.mvs_fuse(s["ctx"].h, s["views"], s["points"], s["src"], s["keep"])
        return n, s["points"], s["src"]
    if kind == "sparse_range":
        mvs.mvs_sparse_depth_range(s["ctx"].h, 0, s["X"], s["vis"], s["reproj"], s["obs"], s["range"], d_lo=D_LO,
                                   d_hi=D_HI)
        return s["range"]
    if kind == "propose":
        img, plane, cost, _, _ = s["inputs"]
        mvs.mvs_cnn_propose(s["net"].h, img, plane, cost, s["Kinv"], s["proposals"])
        return s["proposals"]
    loss = mvs.mvs_cnn_backward(s["net"].h, *s["inputs"])
    return loss, mvs.mvs_cnn_get_grads(s["net"].h)


def work(case):
    kind, px = case["kind"], case["W"] * case["H"]
    # one bilinear window sample: homography, division, three lerps, moments
    per_sample = 26
    if kind in ("depth", "plane_cost", "plane_infer"):
        n, win = case["n_src"], case["samples"] ** 2
        images = px * (n + 1)
        if kind == "plane_cost":
            return {"bytes": images + px * (16 + 4 + 4 * n), "flops": per_sample * win * n * px}
        if kind == "plane_infer":
            # a fifth to a quarter of the pixels are holes with up to four hypotheses
            return {"bytes": images + px * (16 + 4 + 16), "flops": per_sample * win * n * 0.25 * 4 * px}
        # per iteration: three refined planes, one new neighbour's, the proposals
        # once; without a given state also the first plane. Two thirds of the
        # (plane, view) pairs fall inside the sources.
        planes = case["iters"] * 4 + (case["n_prop"] or 1)
        return {"bytes": images + px * (20 + 16 * case["n_prop"]), "flops": per_sample * win * n * 0.66 * planes * px}
    if kind == "batch":
        px = sum(w * h for w, h in _view_sizes(case))
        n = case["n_views"] - 1
        return {"bytes": px + 20 * px,
                "flops": per_sample * case["samples"] ** 2 * n * 0.66 * (case["iters"] * 4 + 1) * px}
    if kind == "geo_filter":
        return {"bytes": px * 16 * (1 + case["n_src"]) + 5 * px, "flops": 100 * case["n_src"] * px}
    if kind == "fuse":
        px = sum(w * h for w, h in _view_sizes(case))
        return {"bytes": px * (16 + 1) + px // 4 * 24, "flops": 60 * case["n_views"] / 2 * px}
    if kind == "sparse_range":
        # the points of the disc of radius W / 10 around each pixel
        near = case["points"] * min(1.0, math.pi * (case["W"] / 10.0) ** 2 / px)
        return {"bytes": px * 8 + case["points"] * 56, "flops": 5 * near * px}
    flops = proposals.cnn_flops(case["W"], case["H"])
    if kind == "propose":
        return {"bytes": px * (1 + 16 + 4 + 64), "flops": flops}
    return {"bytes": px * (1 + 16 + 4 + 16 + 1), "flops": 3 * flops}


# ---------------------------------------------------------------------------
# the same numbers in 64 bits
# ---------------------------------------------------------------------------
def _exact_plane_cost(case, seed):
    """Per-view costs 1 - ZNCC and their weighted mean of a given plane map."""
    g = _generator(seed)
    W, H, n_src, n = case["W"], case["H"], case["n_src"], case["samples"]
    sc = _Scene(seed, [(W, H)] * (1 + n_src), (15.0, 40.0))
    views = [sc.view(v) for v in range(1 + n_src)]
    plane = _estimated(views[0][1], views[0][2], g, wrong=0.3)[0].double()
    imgs = [v[0].double() / 255.0 for v in views]
    K, R0, t0 = sc.cams[0]
    Kinv = torch.as_tensor(np.linalg.inv(K), device=DEV)
    step = case["radius"] / (0.5 * (n - 1))
    off = step * (torch.arange(n, device=DEV, dtype=torch.float64) - 0.5 * (n - 1))
    ov, ou = (a.reshape(-1) for a in torch.meshgrid(off, off, indexing="ij"))

    def bilinear(img, u, v):
        u, v = u.clamp(0, W - 1), v.clamp(0, H - 1)
        x, y = u.floor().clamp(max=W - 2), v.floor().clamp(max=H - 2)
        a, b = u - x, v - y
        i = (y * W + x).long()
        p = img.reshape(-1)
        return (1 - b) * ((1 - a) * p[i] + a * p[i + 1]) + b * ((1 - a) * p[i + W] + a * p[i + W + 1])

    cost = torch.empty(H * W, dtype=torch.float64, device=DEV)
    view_cost = torch.empty((H * W, n_src), dtype=torch.float64, device=DEV)
    for at in torch.arange(H * W, device=DEV).split(1 << 17):
        x, y = (at % W).double(), (at // W).double()
        u, v = x[:, None] + ou, y[:, None] + ov
        inside = (u >= 0) & (u <= W - 1) & (v >= 0) & (v <= H - 1)
        ref = bilinear(imgs[0], u, v)
        centre = imgs[0].reshape(-1)[at][:, None]
        w = torch.exp(-(ou ** 2 + ov ** 2) / (2 * 5.0 ** 2) - (ref - centre) ** 2 / (2 * 0.2 ** 2)) * inside
        ws = w.sum(1, keepdim=True)
        dr = ref - (w * ref).sum(1, keepdim=True) / ws
        vr = (w * dr * dr).sum(1) / ws[:, 0]
        nrm, d = plane.reshape(-1, 4)[at, :3], plane.reshape(-1, 4)[at, 3]
        ray = torch.stack([x, y, torch.ones_like(x)], 1) @ Kinv.T
        rho = d * (nrm * ray).sum(1)
        m = (nrm @ Kinv) / rho[:, None]
        # the plane faces the camera at the pixel and at every sample
        front = (u[..., None] * (nrm @ Kinv)[:, None, 0:1])[..., 0] + v * (nrm @ Kinv)[:, 1:2] + (nrm @ Kinv)[:, 2:3]
        usable = ((nrm * ray).sum(1) < -1e-3 * ray.norm(dim=1)) & ((front < 0) | ~inside).all(1) & (vr >= 1e-6)
        num = torch.zeros_like(x)
        den = torch.zeros_like(x)
        for j in range(n_src):
            Kj, Rj, tj = sc.cams[1 + j]
            A = torch.as_tensor(Kj @ Rj @ R0.T @ np.linalg.inv(K), device=DEV)
            b = torch.as_tensor(Kj @ (tj - Rj @ R0.T @ t0), device=DEV)
            mx = m[:, 0:1] * u + m[:, 1:2] * v + m[:, 2:3]
            q = [A[k, 0] * u + A[k, 1] * v + A[k, 2] + b[k] * mx for k in range(3)]
            us, vs = q[0] / q[2], q[1] / q[2]
            seen = ((q[2] > 0) & (us >= 0) & (us <= W - 1) & (vs >= 0) & (vs <= H - 1)) | ~inside
            ok = usable & seen.all(1)
            src = bilinear(imgs[1 + j], torch.nan_to_num(us), torch.nan_to_num(vs))
            ds = src - (w * src).sum(1, keepdim=True) / ws
            var = (w * ds * ds).sum(1) / ws[:, 0]
            z = (w * dr * ds).sum(1) / ws[:, 0] / torch.sqrt(vr * var)
            c = torch.where(ok & (var >= 1e-6), 1.0 - z.clamp(-1, 1), torch.tensor(2.0, dtype=torch.float64, device=DEV))
            view_cost[at, j] = c
            used = c < 2.0
            num += used
            den += torch.where(used, 1.0 / c.clamp(min=1e-6), torch.zeros_like(c))
        cost[at] = torch.where(num > 0, num / den.clamp(min=1e-300), torch.full_like(num, 2.0))
    return cost.reshape(H, W), view_cost.reshape(H, W, n_src)


def _exact_sparse(case, seed):
    g = _generator(seed)
    W, H = case["W"], case["H"]
    sc = _Scene(seed, [(W, H)] * (1 + case["n_src"]), (15.0, 40.0))
    views = [sc.view(v, image=False) for v in range(len(sc.sizes))]
    _noise_images(sc, g)
    s = _sparse(sc, views, case["points"], g)
    seen_by = sum((s["vis"] >> v) & 1 for v in range(len(views)))
    least = math.floor(float(seen_by.double().mean()) - 1.0)
    use = ((s["vis"] & 1) == 1) & (s["reproj"] < 2.0) & (seen_by >= least)
    p, z = s["obs"][use], s["X"][use][:, 2]
    out = torch.empty((H * W, 2), dtype=torch.float64, device=DEV)
    for at in torch.arange(H * W, device=DEV).split(1 << 14):
        dx, dy = p[None, :, 0] - (at % W)[:, None], p[None, :, 1] - (at // W)[:, None]
        d2 = dx * dx + dy * dy
        near = d2 < (W / 10.0) ** 2
        right, below = dx >= 0, dy >= 0
        lo = torch.full((len(at),), math.inf, dtype=torch.float64, device=DEV)
        hi = -lo
        for quadrant in (right & below, ~right & below, ~right & ~below, right & ~below):
            best, k = torch.where(quadrant & near, d2, math.inf).min(1)
            got = torch.isfinite(best)
            lo = torch.where(got, torch.minimum(lo, z[k]), lo)
            hi = torch.where(got, torch.maximum(hi, z[k]), hi)
        none = lo > hi
        r = torch.stack([lo, hi], 1).clamp(D_LO, D_HI)
        out[at] = torch.where(none[:, None], torch.tensor(math.nan, dtype=torch.float64, device=DEV), r)
    return out.reshape(H, W, 2)


# (input channels, output channels) of the encoder, the decoder and the head
_ENC = ((16, 32), (32, 48), (48, 64), (64, 96), (96, 128))
_DEC = ((224, 96), (160, 64), (112, 48), (80, 32))


def _exact_net(case, seed, train):
    g = _generator(seed)
    W, H = case["W"], case["H"]
    sc = _Scene(seed, [(W, H)], (15.0, 40.0))
    img, plane, cost, target, mask = _net_inputs(sc, g)
    theta = torch.as_tensor(np.load(proposals.WEIGHTS), dtype=torch.float64, device=DEV).requires_grad_(train)
    at = 0

    def conv(x, ci, co, k):
        nonlocal at
        w = theta[at:at + co * k * k * ci].reshape(co, k, k, ci).permute(0, 3, 1, 2)
        at += co * k * k * ci
        b = theta[at:at + co]
        at += co
        # as a matrix product per tap
        xp = torch.nn.functional.pad(x, (k // 2,) * 4)
        y = b[:, None, None].expand(co, x.shape[1], x.shape[2])
        for t in range(k * k):
            part = xp[:, t // k:t // k + x.shape[1], t % k:t % k + x.shape[2]]
            y = y + (w[:, :, t // k, t % k] @ part.reshape(ci, -1)).reshape(y.shape)
        return y

    rho_lo, rho_hi = 1.0 / D_HI, 1.0 / D_LO
    p = plane.double()
    x = torch.zeros((16, H, W), dtype=torch.float64, device=DEV)
    x[0] = img.double() / 255.0
    x[1] = (1.0 / p[..., 3] - rho_lo) / (rho_hi - rho_lo)
    x[2:5] = p[..., :3].permute(2, 0, 1)
    x[5] = cost.double() * 0.5
    with torch.set_grad_enabled(train):
        skip = []
        for ci, co in _ENC:
            if skip:
                x = torch.nn.functional.avg_pool2d(x[None], 2)[0]
            x = torch.relu(conv(x, ci, co, 3))
            skip.append(x)
        for level, (ci, co) in zip((3, 2, 1, 0), _DEC):
            up = x.repeat_interleave(2, 1).repeat_interleave(2, 2)
            x = torch.relu(conv(torch.cat([up, skip[level]]), ci, co, 3))
        y = conv(x, 32, 16, 1).reshape(4, 4, H, W)
        rho = rho_lo + (rho_hi - rho_lo) * torch.sigmoid(y[:, 0])
        n = y[:, 1:] / y[:, 1:].norm(dim=1, keepdim=True)
        if train:
            t = target.double()
            l = ((rho - 1.0 / t[..., 3]).abs() / (rho_hi - rho_lo) +
                 0.1 * (1.0 - (n * t[..., :3].permute(2, 0, 1)).sum(1).abs()))
            loss = (l.min(0).values * mask).sum() / (W * H)
            return loss.item(), torch.autograd.grad(loss, theta)[0]
    K = sc.cams[0][0]
    yy, xx = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float64),
                            torch.arange(W, device=DEV, dtype=torch.float64), indexing="ij")
    ray = torch.stack([(xx - K[0, 2]) / K[0, 0], (yy - K[1, 2]) / K[1, 1], torch.ones_like(xx)])
    n = torch.where((n * ray).sum(1, keepdim=True) > 0, -n, n)
    return torch.cat([n, 1.0 / rho[:, None]], 1).permute(2, 3, 0, 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "plane_cost":
        return _exact_plane_cost(case, seed)
    if kind == "sparse_range":
        return _exact_sparse(case, seed)
    if kind == "propose":
        return _exact_net(case, seed, False)
    if kind == "train":
        return _exact_net(case, seed, True)
    # depth maps, filled maps, masks and fused points follow from comparisons
    # of costs and positions: in 64 bits other candidates win near a tie
    return None
