"""A PatchMatch call captured into the caller's own CUDA graph stays valid while
later calls of the context need a larger workspace or give it back."""
import copy

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stored", [True, False])
def test_replay_after_the_workspace_has_grown(mvs_lib, stored):
    import torch
    from paper_2104_06165_gb300 import scenes
    sc, srcs = scenes.scene_batch(seed=5, sizes=((60, 40), (90, 61), (48, 33)), n_src=2)
    stream = torch.cuda.Stream()
    p = mvs_lib.PMParams(win_radius=5.0, win_samples=6, iters=2, seed=11)
    out = [(torch.zeros((h, w, 4), device="cuda"), torch.zeros((h, w), device="cuda"))
           for h, w in ((im.shape) for im in sc.images)]
    torch.cuda.synchronize()
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=stream) as ctx:
        if not stored:
            mvs_lib.mvs_window_limit(ctx.h, 0)
        mvs_lib.mvs_patchmatch(ctx.h, 0, srcs[0], p, *out[0])
        torch.cuda.synchronize()
        first = [t.cpu().numpy() for t in out[0]]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            mvs_lib.mvs_patchmatch(ctx.h, 0, srcs[0], p, *out[0])
        # a larger view and a larger window; then what there is goes back
        wide = copy.copy(p)
        wide.win_samples, wide.win_radius = 21, 10.0
        mvs_lib.mvs_window_limit(ctx.h, 1 << 34)
        mvs_lib.mvs_patchmatch(ctx.h, 1, srcs[1], wide, *out[1])
        mvs_lib.mvs_window_limit(ctx.h, 0)
        torch.cuda.synchronize()
        for t in out[0]:
            t.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert all(np.array_equal(t.cpu().numpy(), f) for t, f in zip(out[0], first))
        mvs_lib.mvs_patchmatch(ctx.h, 0, srcs[0], p, *out[0])
        torch.cuda.synchronize()
        assert all(np.array_equal(t.cpu().numpy(), f) for t, f in zip(out[0], first))
