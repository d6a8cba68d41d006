"""The sparse depth ranges on both sides of the rule that chooses between
scanning every feature and searching cells, with cells of the smallest side
(16 pixels), a few tiles' side and the side that the radius allows, against
the stated rule over all features (single-precision distances, every
operation rounded on its own, the first feature winning a tie): bit for bit.
A feature without a depth takes part in neither."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _all_features(W, H, u, v, z):
    """In float32 on the device; separate operations, so nothing contracts."""
    import torch
    u, v, z = (torch.from_numpy(np.asarray(a, np.float32)).cuda() for a in (u, v, z))
    r = np.float32(W) / np.float32(10.0)
    r2, inf = float(r * r), float("inf")
    out = torch.full((H, W, 2), float("nan"), device="cuda")
    dx = u[None, :] - torch.arange(W, device="cuda", dtype=torch.float32)[:, None]
    first = torch.arange(len(z), device="cuda")
    for y in range(H):
        dy = (v - float(y))[None, :]
        d2 = dx * dx + dy * dy
        lo = torch.full((W,), inf, device="cuda")
        hi = -lo
        for q in ((dx >= 0) & (dy >= 0), (dx < 0) & (dy >= 0), (dx < 0) & (dy < 0), (dx >= 0) & (dy < 0)):
            d = torch.where(q & (d2 < r2), d2, inf)
            m = d.amin(1)
            k = torch.where(d == m[:, None], first, len(z)).amin(1)
            got = torch.isfinite(m)
            zk = z[k]
            lo = torch.where(got, torch.minimum(lo, zk), lo)
            hi = torch.where(got, torch.maximum(hi, zk), hi)
        ok = lo <= hi
        out[y, ok, 0] = lo[ok].clamp(2.0, 8.0)
        out[y, ok, 1] = hi[ok].clamp(2.0, 8.0)
    return out.cpu().numpy()


@pytest.mark.parametrize("W, H, n", [
    (608, 256, 9000),                       # 608 tiles: scanned
    (609, 256, 9000),                       # 624: cells of 16 pixels
    (1600, 800, 1000), (1600, 800, 1001),   # 5000 tiles: scanned; cells of 64 pixels
    (3001, 500, 1100),                      # 6016 tiles, ragged: cells of 64 pixels
    (160, 16000, 1100),                     # 10000 tiles, few points nearby: the radius' 32 pixels
])
def test_ranges_on_both_sides_of_the_rule(mvs_lib, W, H, n):
    import torch
    rng = np.random.default_rng(W + n)
    obs = np.stack([rng.uniform(-0.05 * W, 1.05 * W, n), rng.uniform(-0.05 * H, 1.05 * H, n)], 1)
    obs[::4] = np.round(obs[::4])
    obs[1::9] = 16.0 * np.round(obs[1::9] / 16.0)
    z = rng.uniform(1.5, 8.5, n)
    z[2::7] = np.nan
    X = np.stack([np.zeros(n), np.zeros(n), z], 1)
    vis = np.full(n, 3, np.uint64)
    rep = np.where(rng.random(n) < 0.1, 5.0, 0.1)
    K = np.array([[W, 0.0, W / 2.0], [0.0, W, H / 2.0], [0.0, 0.0, 1.0]])
    images = [np.zeros((H, W), np.uint8), np.zeros((48, 64), np.uint8)]
    out = np.zeros((H, W, 2), np.float32)
    with mvs_lib.Context([K, K], [np.eye(3)] * 2, [np.zeros(3), np.array([1.0, 0.0, 0.0])], images,
                         stream=torch.cuda.current_stream()) as ctx:
        mvs_lib.mvs_sparse_depth_range(ctx.h, 0, X, vis, rep, obs, out)
    use = (rep < 2.0) & (z == z)
    assert np.array_equal(out, _all_features(W, H, obs[use, 0], obs[use, 1], z[use]), equal_nan=True)
