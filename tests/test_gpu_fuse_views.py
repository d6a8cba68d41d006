"""Fusion where the claim pass's record of agreeing views runs out of bits
(more than 32 later views) and where one block, or one pixel row, holds a
view: a plane seen by cameras shifted by whole pixels, whose projections are
exact, against the FP64 oracle point for point."""
import numpy as np
import pytest

from test_gpu_fusion import _close, _load_maps

pytestmark = pytest.mark.gpu

F, D, B = 100.0, 4.0, 0.2      # a shift of F B / D = 5 pixels


@pytest.mark.parametrize("n, W, H", [(2, 7, 3), (5, 24, 8), (34, 200, 3), (45, 260, 2)])
def test_many_shifted_views_equal_the_oracle(mvs_lib, oracle_lib, n, W, H):
    import torch
    rng = np.random.default_rng(n)
    K = np.tile(np.array([[F, 0, 0.5 * (W - 1)], [0, F, 0.5 * (H - 1)], [0, 0, 1]]), (n, 1, 1))
    R = np.tile(np.eye(3), (n, 1, 1))
    t = np.array([[-k * B, 0.0, 0.0] for k in range(n)])
    imgs = [np.full((H, W), 128, np.uint8) for _ in range(n)]
    pl = np.zeros((H, W, 4))
    pl[..., 2], pl[..., 3] = -1.0, D
    maps = {v: pl for v in range(n)}
    order = [int(v) for v in rng.permutation(n)]
    keep = {v: (rng.random((H, W)) < 0.9).astype(np.uint8) for v in range(n)}
    cap = n * W * H
    pts, src = np.zeros((cap, 4), np.float32), np.zeros((cap, 2), np.int32)
    with mvs_lib.Context(K, R, t, imgs, stream=torch.cuda.current_stream()) as ctx:
        _load_maps(mvs_lib, ctx, maps, n)
        m = mvs_lib.mvs_fuse(ctx.h, order, pts, src, keep_masks=[keep[v] for v in order])
    opts, osv, osp = oracle_lib.fuse(oracle_lib.Scene(K, R, t, imgs), order, maps, keep=keep)
    assert m == len(opts) and opts[:, 3].max() > (32 if n > 33 else 1)
    assert np.array_equal(src[:m, 0], osv) and np.array_equal(src[:m, 1], osp)
    assert _close(pts[:m], opts)
