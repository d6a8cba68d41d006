"""A wait of the message passing that runs out: no node gets a label, the map
stays, the status is reported once, by the call itself with host
buffers and with device buffers by the next call that would use the result, and
the call after that works."""
import numpy as np
import pytest

from test_gpu_trw import _inputs

pytestmark = pytest.mark.gpu


def _gives_up(mvs, call):
    with pytest.raises(mvs.MvsError) as e:
        call()
    assert e.value.status == mvs.MVS_ETIMEOUT


@pytest.mark.parametrize("W, H, iters", [(64, 64, 1), (130, 300, 3)])
def test_labels_say_nothing(mvs_lib, W, H, iters):
    import torch
    from paper_2104_06165_gb300 import scenes
    sc = scenes.make_scene(W=16, H=16, n_src=1, seed=1)
    args = _inputs(W, H, 0.6, 3)
    shape = ((H + 1) // 2, (W + 1) // 2)
    phi = mvs_lib.PhiParams(trw_iters=iters)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        ref = np.zeros(shape, np.int32)
        mvs_lib.mvs_phi_mrf(ctx.h, *args, phi, ref)
        # host buffers
        mvs_lib.mvs_phi_test_timeout(ctx.h)
        label = np.full(shape, -7, np.int32)
        _gives_up(mvs_lib, lambda: mvs_lib.mvs_phi_mrf(ctx.h, *args, phi, label))
        assert (label == -2).all()
        mvs_lib.mvs_phi_mrf(ctx.h, *args, phi, label)
        assert np.array_equal(label, ref)
        # device buffers
        dev = [torch.from_numpy(a).cuda() for a in args]
        out = torch.full(shape, -7, dtype=torch.int32, device="cuda")
        mvs_lib.mvs_phi_test_timeout(ctx.h)
        mvs_lib.mvs_phi_mrf(ctx.h, *dev, phi, out)
        torch.cuda.synchronize()
        _gives_up(mvs_lib, lambda: mvs_lib.mvs_phi_mrf(ctx.h, *dev, phi, out))
        torch.cuda.synchronize()
        assert (out == -2).all()
        mvs_lib.mvs_phi_mrf(ctx.h, *dev, phi, out)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), ref)


def test_map_stays_and_whoever_reads_it_is_told(mvs_lib):
    import torch
    from paper_2104_06165_gb300 import scenes
    W, H = 96, 72
    sc = scenes.make_scene(W=W, H=H, n_src=3, seed=5, baseline_frac=0.1)
    srcs = [1, 2, 3]
    p = mvs_lib.PMParams(win_radius=5.0, win_samples=6, iters=2, seed=3)
    phi = mvs_lib.PhiParams(trw_iters=2)
    rng = np.random.default_rng(2)
    keep = (rng.random((H, W)) < 0.4).astype(np.uint8)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        plane, cost = np.zeros((H, W, 4), np.float32), np.zeros((H, W), np.float32)
        mvs_lib.mvs_patchmatch(ctx.h, 0, srcs, p, plane, cost)
        for v in srcs:
            mvs_lib.mvs_set_depth_map(ctx.h, v, plane, cost)
        filled = plane.copy()
        mvs_lib.mvs_plane_infer(ctx.h, 0, srcs, p, phi, keep, filled, cost)
        assert not np.array_equal(filled, plane)
        # host buffers: the given map stays, in the caller's buffer and in the context
        mvs_lib.mvs_set_depth_map(ctx.h, 0, plane, cost)
        points = np.zeros((4 * W * H, 4), np.float32)
        fused = mvs_lib.mvs_fuse(ctx.h, [0, 1, 2, 3], points)
        again = plane.copy()
        mvs_lib.mvs_phi_test_timeout(ctx.h)
        _gives_up(mvs_lib, lambda: mvs_lib.mvs_plane_infer(ctx.h, 0, srcs, p, phi, keep, again, cost))
        assert np.array_equal(again, plane)
        other = np.zeros_like(points)
        assert mvs_lib.mvs_fuse(ctx.h, [0, 1, 2, 3], other) == fused and np.array_equal(other, points)
        # device buffers: fusion, filter and inference are told, once
        d_plane, d_cost, d_keep = (torch.from_numpy(a).cuda() for a in (plane, cost, keep))
        mask = np.zeros((H, W), np.uint8)
        for told in (lambda: mvs_lib.mvs_fuse(ctx.h, [0, 1], other),
                     lambda: mvs_lib.mvs_geo_filter(ctx.h, 0, srcs, mvs_lib.FilterParams(), mask),
                     lambda: mvs_lib.mvs_plane_infer(ctx.h, 0, srcs, p, phi, d_keep, d_plane, d_cost)):
            mvs_lib.mvs_phi_test_timeout(ctx.h)
            mvs_lib.mvs_plane_infer(ctx.h, 0, srcs, p, phi, d_keep, d_plane, d_cost)
            torch.cuda.synchronize()      # (a call that only enqueues checks when it is made)
            _gives_up(mvs_lib, told)
            assert np.array_equal(d_plane.cpu().numpy(), plane)
            told_again = mvs_lib.mvs_fuse(ctx.h, [0, 1], other)
            assert told_again > 0
        mvs_lib.mvs_plane_infer(ctx.h, 0, srcs, p, phi, d_keep, d_plane, d_cost)
        torch.cuda.synchronize()
        assert np.array_equal(d_plane.cpu().numpy(), filled)
