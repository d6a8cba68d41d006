"""Stored and rebuilt windows, and the work layouts of every window size.

A call of several iterations stores each pixel's window once and reads it
back (k_phase<..., STORED>); a call of one phase on a given state rebuilds
it.  Both evaluate the same expressions, so the maps are equal bit for bit,
at sizes where the 1 x 8 tiles, the super-tiles and the borders are ragged.
"""
import copy

import numpy as np
import pytest

from test_gpu_bench_layout import _check_costs

pytestmark = pytest.mark.gpu

# one window size on each side of every layout's limit (samples^2 <= 16, 36,
# 64, 128, 176, 256, 320, 384, 448, 484)
LAYOUTS = [4, 5, 6, 8, 9, 11, 12, 13, 14, 16, 17, 18, 19, 20, 21, 22]


def _scene(W, H, n_src, seed):
    from paper_2104_06165_gb300 import scenes
    return scenes.make_scene(W=W, H=H, n_src=n_src, seed=seed, baseline_frac=0.1)


def _maps(H, W):
    return np.zeros((H, W, 4), np.float32), np.zeros((H, W), np.float32)


def _one_call_and_phase_by_phase(mvs, ctx, srcs, p):
    H, W = ctx.shapes[0]
    a = _maps(H, W)
    mvs.mvs_patchmatch(ctx.h, 0, srcs, p, *a)
    b = _maps(H, W)
    q = copy.copy(p)
    q.iters = q.phase_begin = q.phase_end = 0
    mvs.mvs_patchmatch(ctx.h, 0, srcs, q, *b)
    for ph in range(2 * p.iters):
        q = copy.copy(p)
        q.phase_begin, q.phase_end, q.init_mode = ph, ph + 1, mvs.MVS_INIT_GIVEN
        mvs.mvs_patchmatch(ctx.h, 0, srcs, q, *b)
    return a, b


@pytest.mark.parametrize("n", LAYOUTS)
@pytest.mark.parametrize("precision", [0, 1])
def test_stored_windows_equal_rebuilt_ones(mvs_lib, n, precision):
    import torch
    sc = _scene(70, 49, 3, 11)
    p = mvs_lib.PMParams(win_radius=max(2.0, 0.5 * (n - 1)), win_samples=n, iters=2, seed=5, precision=precision)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        a, b = _one_call_and_phase_by_phase(mvs_lib, ctx, [1, 2, 3], p)
        # the initial state given: the windows come from their own kernel
        c = _maps(*ctx.shapes[0])
        q = copy.copy(p)
        q.iters = 0
        mvs_lib.mvs_patchmatch(ctx.h, 0, [1, 2, 3], q, *c)
        q.iters, q.init_mode = 2, mvs_lib.MVS_INIT_GIVEN
        mvs_lib.mvs_patchmatch(ctx.h, 0, [1, 2, 3], q, *c)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    assert np.array_equal(a[0], c[0]) and np.array_equal(a[1], c[1])


@pytest.mark.parametrize("lanes, n", [(8, 6), (16, 8), (8, 11), (32, 11), (32, 15)])
def test_stored_windows_follow_the_lane_hint(mvs_lib, lanes, n):
    import torch
    sc = _scene(70, 49, 3, 12)
    p = mvs_lib.PMParams(win_radius=5.0, win_samples=n, iters=2, seed=6, lanes_per_pixel=lanes)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        a, b = _one_call_and_phase_by_phase(mvs_lib, ctx, [1, 2, 3], p)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("W, H", [(2, 2), (3, 9), (17, 8), (33, 258), (131, 257)])
def test_every_pixel_is_visited_at_ragged_sizes(mvs_lib, W, H):
    """Tiles and super-tiles cut by the border: one call equals phase-by-phase
    calls, and every pixel that can be scored has been refined."""
    import torch
    sc = _scene(W, H, 2, 13)
    p = mvs_lib.PMParams(win_radius=5.0, win_samples=6, iters=3, seed=7)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        a, b = _one_call_and_phase_by_phase(mvs_lib, ctx, [1, 2], p)
        q = copy.copy(p)
        q.iters = 0
        c = _maps(H, W)
        mvs_lib.mvs_patchmatch(ctx.h, 0, [1, 2], q, *c)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    if W * H > 1000:
        assert ((a[0] != c[0]).any(-1))[a[1] < 2.0].mean() > 0.9


def test_workspace_shared_by_views_of_different_size(mvs_lib):
    """One context, views of different sizes and windows in turn (the
    workspace grows and is reused), batched and one by one: equal maps."""
    import torch
    from paper_2104_06165_gb300 import scenes
    sc, srcs = scenes.scene_batch(seed=3, sizes=((60, 40), (90, 61), (48, 33)), n_src=2)
    p = mvs_lib.PMParams(win_radius=5.0, win_samples=6, iters=2, seed=9)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        def batch(par):
            out = [_maps(h, w) for h, w in ctx.shapes]
            mvs_lib.mvs_patchmatch_batch(ctx.h, [0, 1, 2], srcs, par, [o[0] for o in out], [o[1] for o in out])
            return out
        first = batch(p)
        wide = copy.copy(p)
        wide.win_samples, wide.win_radius = 21, 10.0
        for v in (0, 1, 2):           # a larger record: the workspace moves
            mvs_lib.mvs_patchmatch(ctx.h, v, srcs[v], wide, *_maps(*ctx.shapes[v]))
        again = batch(p)              # the captured graph must not keep the old one
        for v in (0, 1, 2):
            one = _maps(*ctx.shapes[v])
            mvs_lib.mvs_patchmatch(ctx.h, v, srcs[v], p, *one)
            for k in (0, 1):
                assert np.array_equal(first[v][k], one[k]) and np.array_equal(again[v][k], one[k])


@pytest.mark.parametrize("n", [12, 13, 17, 18, 20, 22])
def test_costs_of_the_dense_layouts_against_the_oracle(mvs_lib, oracle_lib, n):
    import torch
    sc = _scene(96, 72, 4, 7)
    srcs = [1, 2, 3, 4]
    p = mvs_lib.PMParams(win_radius=0.5 * (n - 1), win_samples=n, iters=0, seed=3)
    osc = oracle_lib.Scene(sc.K, sc.R, sc.t, sc.images)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        pl, co = _maps(72, 96)
        mvs_lib.mvs_patchmatch(ctx.h, 0, srcs, p, pl, co)
        _check_costs(mvs_lib, oracle_lib, ctx, osc, srcs, p, pl, co, np.ones(co.shape, bool), f"{n}x{n}")
