"""The limit on the stored windows: with none, some and all of the views' windows
stored, one call and a batch of uneven views give the same maps bit for bit, and
a batch captured before the limit changed is not replayed over memory that went
back."""
import copy

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _maps(H, W):
    return np.zeros((H, W, 4), np.float32), np.zeros((H, W), np.float32)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("given", [False, True])
def test_maps_do_not_depend_on_the_limit(mvs_lib, precision, given):
    import torch
    from paper_2104_06165_gb300 import scenes
    sc, srcs = scenes.scene_batch(seed=4, sizes=((60, 40), (90, 61), (48, 33)), n_src=2)
    p = mvs_lib.PMParams(win_radius=5.0, win_samples=6, iters=2, seed=10, precision=precision)
    start = copy.copy(p)
    start.iters = 0
    if given:
        p.init_mode = mvs_lib.MVS_INIT_GIVEN
    record = 4 * (2 * 4 * 9 + 16)          # bytes of a 6 x 6 window in 4 x 9 slots
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        first = [_maps(*s) for s in ctx.shapes]
        for v in (0, 1, 2):
            mvs_lib.mvs_patchmatch(ctx.h, v, srcs[v], start, *first[v])

        def run():
            a = [[m.copy() for m in f] for f in first]
            mvs_lib.mvs_patchmatch_batch(ctx.h, [0, 1, 2], srcs, p, [m[0] for m in a], [m[1] for m in a])
            b = [[m.copy() for m in f] for f in first]
            for v in (0, 1, 2):
                mvs_lib.mvs_patchmatch(ctx.h, v, srcs[v], p, *b[v])
            return a + b
        out = []
        # all stored; none; those of the smaller two views only; all again
        for limit in (1 << 34, 0, record * 60 * 40, 1 << 34):
            mvs_lib.mvs_window_limit(ctx.h, limit)
            out += [run(), run()]
        with pytest.raises(mvs_lib.MvsError) as e:
            mvs_lib.mvs_window_limit(ctx.h, -1)
        assert e.value.status == mvs_lib.MVS_EINVAL
    for o in out[1:]:
        for x, y in zip(o, out[0]):
            assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])
    for a, b in zip(out[0][:3], out[0][3:]):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
