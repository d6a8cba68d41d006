"""The cells of the sparse depth ranges against the FP64 oracle, with host and
device buffers, at sizes and densities that the rule sends to them (more than
608 tiles, more than 1000 points, more than 5 M pairs): cells of one and of
several tiles, ragged grids, images narrower than a cell's neighbourhood,
features on cell borders, at equal distances and far outside the image."""
import numpy as np
import pytest

from test_gpu_sparse_rule import _all_features

pytestmark = pytest.mark.gpu

BAND_PX = 1e-4      # as in the stage's parity test


@pytest.mark.parametrize("W, H, n, spread", [
    (656, 250, 8000, 0.3),      # cells of 16 pixels
    (401, 400, 8000, 0.3),      # ragged last cells on both sides
    (97, 1700, 8000, 0.3),      # 7 cells wide; the radius is less than a cell
    (1205, 323, 4000, 0.05),    # cells of 16 pixels, few to a cell
    (2000, 200, 3100, 1.0),     # most features far outside
    (2003, 1001, 1100, 0.05),   # cells of 80 pixels
])
def test_cells_follow_the_oracle(mvs_lib, oracle_lib, W, H, n, spread):
    import torch
    rng = np.random.default_rng(W + n)
    obs = np.stack([rng.uniform(-spread * W, (1 + spread) * W, n), rng.uniform(-spread * H, (1 + spread) * H, n)], 1)
    obs[::4] = np.round(obs[::4])                    # equal distances
    obs[1::9] = 16.0 * np.round(obs[1::9] / 16.0)    # cell borders
    obs[5] = (-1e7, 3e9)                             # beyond any cell arithmetic
    z = rng.uniform(2.0, 8.0, n)
    X = np.stack([np.zeros(n), np.zeros(n), z], 1)   # the reference camera sits at the origin
    vis = np.full(n, 3, np.uint64)
    rep = np.where(rng.random(n) < 0.1, 5.0, 0.1)    # some features are not used
    K = np.array([[W, 0.0, W / 2.0], [0.0, W, H / 2.0], [0.0, 0.0, 1.0]])
    images = [np.zeros((H, W), np.uint8), np.zeros((48, 64), np.uint8)]
    out = np.zeros((H, W, 2), np.float32)
    with mvs_lib.Context([K, K], [np.eye(3)] * 2, [np.zeros(3), np.array([1.0, 0.0, 0.0])], images,
                         stream=torch.cuda.current_stream()) as ctx:
        mvs_lib.mvs_profile(ctx.h, False)
        mvs_lib.mvs_sparse_depth_range(ctx.h, 0, X, vis, rep, obs, out)
        # count, features, scan, fill and search; the scan of every feature takes three
        assert mvs_lib.mvs_profile_read(ctx.h)[2] == 5
        dev = torch.zeros((H, W, 2), device="cuda")
        mvs_lib.mvs_sparse_depth_range(ctx.h, 0, torch.from_numpy(X).cuda(), torch.from_numpy(vis.view(np.int64)).cuda(),
                                       torch.from_numpy(rep).cuda(), torch.from_numpy(obs).cuda(), dev)
        assert np.array_equal(dev.cpu().numpy(), out, equal_nan=True)
    use = rep < 2.0
    o, frag = oracle_lib.sparse_range(W, H, obs[use], z[use], d_lo=2.0, d_hi=8.0, band_px=BAND_PX, fragile=True)
    firm = ~frag.astype(bool)
    assert np.array_equal(out[firm], o.astype(np.float32)[firm], equal_nan=True)
    # the rounded features make exact ties, which the oracle calls fragile
    assert np.array_equal(out, _all_features(W, H, obs[use, 0], obs[use, 1], z[use]), equal_nan=True)
