"""Line-fit hypotheses from bit maps at the shapes where the maps change:
words and summaries (32 and 1024 positions) cut by the border, rows against
columns, images so narrow that the diagonals run along x; and plane inference
against its own stages, of which it scores only the MRF's nodes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(mvs_lib):
    import torch
    from paper_2104_06165_gb300 import scenes
    sc = scenes.make_scene(W=16, H=16, n_src=1, seed=1)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as c:
        yield c


@pytest.mark.parametrize("W, H", [(2, 2), (31, 33), (64, 32), (97, 3), (3, 97), (2, 131), (40, 1100), (1100, 40),
                                  (1025, 33), (3, 1030)])
@pytest.mark.parametrize("n_fit, inverse", [(6, 0), (2, 1), (8, 0), (9, 0)])
def test_hypotheses_follow_the_oracle(ctx, mvs_lib, oracle_lib, W, H, n_fit, inverse):
    rng = np.random.default_rng(W * 7 + H)
    yy, xx = np.mgrid[0:H, 0:W]
    depth = 3.0 + 0.001 * xx + 0.0007 * yy
    known = (rng.random((H, W)) < 0.5)
    known &= ((xx // 45 + yy // 45) % 3 != 1)              # blocks of holes
    known[:, W // 2:] &= rng.random((H, W - W // 2)) < 0.01   # and almost empty words
    known = known.astype(np.uint8)
    depth = (depth * known).astype(np.float32)
    hyp = np.zeros((H, W, 4), np.float32)
    valid = np.zeros((H, W, 4), np.uint8)
    phi = mvs_lib.PhiParams(n_fit=n_fit, fit_inverse=inverse)
    mvs_lib.mvs_phi_hypotheses(ctx.h, depth, known, phi, 2.0, 8.0, hyp, valid)
    ohyp, ovalid = oracle_lib.phi_hypotheses(depth.astype(np.float64), known, n_fit=n_fit, inverse=bool(inverse),
                                             d_lo=2.0, d_hi=8.0)
    near_bound = (np.abs(ohyp - 2.0) < 1e-3) | (np.abs(ohyp - 8.0) < 1e-3)
    assert ((valid != ovalid) & ~near_bound).sum() == 0
    both = (valid == 1) & (ovalid == 1)
    if both.any():
        assert (np.abs(hyp - ohyp)[both] / ohyp[both]).max() < 1e-3


@pytest.mark.parametrize("W, H", [(64, 48), (65, 49)])
@pytest.mark.parametrize("selection", [0, 1])
def test_inference_equals_its_stages(mvs_lib, W, H, selection):
    import torch
    from paper_2104_06165_gb300 import scenes
    sc = scenes.make_scene(W=W, H=H, n_src=3, seed=5, baseline_frac=0.1)
    srcs = [1, 2, 3]
    p = mvs_lib.PMParams(win_radius=5.0, win_samples=6, iters=2, seed=3)
    phi = mvs_lib.PhiParams(selection=selection)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as c:
        plane, cost = np.zeros((H, W, 4), np.float32), np.zeros((H, W), np.float32)
        mvs_lib.mvs_patchmatch(c.h, 0, srcs, p, plane, cost)
        whole = plane.copy()
        mvs_lib.mvs_plane_infer(c.h, 0, srcs, p, phi, None, whole, cost)
        known = ((plane[..., 3] > 0) & (cost < phi.hole_cost)).astype(np.uint8)
        depth = np.where(known, plane[..., 3], 0).astype(np.float32)
        hyp, valid = np.zeros((H, W, 4), np.float32), np.zeros((H, W, 4), np.uint8)
        mvs_lib.mvs_phi_hypotheses(c.h, depth, known, phi, p.d_lo, p.d_hi, hyp, valid)
        hcost = np.zeros((H, W, 4), np.float32)
        mvs_lib.mvs_phi_cost(c.h, 0, srcs, p, hyp, valid, hcost)
        parts = plane.copy()
        if selection:
            mvs_lib.mvs_phi_select_min_cost(c.h, 0, known, hyp, valid, hcost, parts)
        else:
            label = np.zeros(((H + 1) // 2, (W + 1) // 2), np.int32)
            mvs_lib.mvs_phi_mrf(c.h, known, depth, hyp, valid, hcost, phi, label)
            mvs_lib.mvs_phi_select(c.h, 0, known, hyp, valid, label, parts)
    assert (known == 0).any() and np.array_equal(whole, parts)
