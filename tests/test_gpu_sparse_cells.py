"""Binned closest-feature search where the cells of 32 pixels and their rings
change: one cell, ragged cells, few and many features, features on cell
borders, outside the image and at equal distances.  Compared with the FP64
oracle at firm choices, and bit for bit with the stated rule evaluated over
all features (distances in single precision, every operation rounded on its
own, the first feature winning a tie)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BAND_PX = 1e-4      # as in the stage's parity test


def _all_features(W, H, obs, z):
    """The rule without bins, in float32."""
    u, v, z = (np.asarray(a, np.float32) for a in (obs[:, 0], obs[:, 1], z))
    if not len(z):
        return np.full((H, W, 2), np.nan, np.float32)
    r = np.float32(W) / np.float32(10.0)
    lo = np.full((H, W), np.inf, np.float32)
    hi = np.full((H, W), -np.inf, np.float32)
    for y in range(H):
        dx = u[None, :] - np.arange(W, dtype=np.float32)[:, None]
        dy = (v - np.float32(y))[None, :]
        d2 = dx * dx + dy * dy
        for q in (dx >= 0) & (dy >= 0), (dx < 0) & (dy >= 0), (dx < 0) & (dy < 0), (dx >= 0) & (dy < 0):
            d = np.where(q & (d2 < r * r), d2, np.float32(np.inf))
            k = d.argmin(1)                        # the first of equal distances
            got = np.isfinite(d[np.arange(W), k])
            lo[y] = np.where(got, np.minimum(lo[y], z[k]), lo[y])
            hi[y] = np.where(got, np.maximum(hi[y], z[k]), hi[y])
    out = np.stack([lo, hi], -1).clip(2.0, 8.0)
    out[lo > hi] = np.nan
    return out


@pytest.mark.parametrize("W, H", [(20, 14), (33, 64), (160, 97), (400, 40)])
@pytest.mark.parametrize("n", [0, 1, 5, 200, 3000])
def test_ranges_follow_the_oracle(mvs_lib, oracle_lib, W, H, n):
    import torch
    from paper_2104_06165_gb300 import scenes
    sc = scenes.make_scene(W=W, H=H, n_src=1, seed=1)
    rng = np.random.default_rng(W + n)
    obs = np.stack([rng.uniform(-0.3 * W, 1.3 * W, n), rng.uniform(-0.3 * H, 1.3 * H, n)], 1)
    obs[::4] = np.round(obs[::4])                  # equal distances, cell borders
    obs[1::9] = 32.0 * np.round(obs[1::9] / 32.0)
    z = rng.uniform(2.0, 8.0, n)
    X = np.stack([np.zeros(n), np.zeros(n), z], 1) # the reference camera sits at the origin
    vis = np.full(n, 3, np.uint64)
    rep = np.where(rng.random(n) < 0.1, 5.0, 0.1)  # some features are not used
    out = np.zeros((H, W, 2), np.float32)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        mvs_lib.mvs_sparse_depth_range(ctx.h, 0, X, vis, rep, obs, out)
        dev = torch.zeros((H, W, 2), device="cuda")
        if n:
            mvs_lib.mvs_sparse_depth_range(ctx.h, 0, torch.from_numpy(X).cuda(), torch.from_numpy(vis.view(np.int64)).cuda(),
                                           torch.from_numpy(rep).cuda(), torch.from_numpy(obs).cuda(), dev)
            assert np.array_equal(dev.cpu().numpy(), out, equal_nan=True)
    if n == 0:
        assert np.isnan(out).all()
        return
    use = rep < 2.0
    o, frag = oracle_lib.sparse_range(W, H, obs[use], z[use], d_lo=2.0, d_hi=8.0, band_px=BAND_PX, fragile=True)
    firm = ~frag.astype(bool)
    o = o.astype(np.float32)
    assert np.array_equal(out[firm], o[firm], equal_nan=True)
    # the rounded features make exact ties, which the oracle calls fragile
    assert np.array_equal(out, _all_features(W, H, obs[use], z[use]), equal_nan=True)
