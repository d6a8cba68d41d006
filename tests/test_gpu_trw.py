"""Row-pipelined message passing (k_trw_rows) against the FP64 oracle at the
sizes where its schedule changes: one row, rows around a block of 8, several
blocks, columns around the 8-column polls, the 32-column chunks and the
128-column ring, with holes from isolated pixels to the whole image."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# the tie band of the belief that the parity test of the stage uses
GAP = 1e-3


def _inputs(W, H, holes, seed):
    rng = np.random.default_rng(seed)
    known = (rng.random((H, W)) >= holes).astype(np.uint8)
    yy, xx = np.mgrid[0:H, 0:W]
    depth = (3.0 + 0.01 * xx + 0.007 * yy).astype(np.float32)
    hyp = (depth[..., None] * (1.0 + rng.uniform(-0.2, 0.2, (H, W, 4)))).astype(np.float32)
    valid = (rng.random((H, W, 4)) < 0.7).astype(np.uint8)   # also holes with one or no hypothesis
    cost = rng.uniform(0.0, 2.0, (H, W, 4)).astype(np.float32)
    return known, (depth * known).astype(np.float32), hyp, valid, cost


@pytest.mark.parametrize("W, H", [(2, 2), (18, 2), (64, 15), (62, 16), (63, 18), (130, 34), (258, 20), (540, 50),
                                  (20, 530)])
@pytest.mark.parametrize("holes", [0.05, 0.5, 1.0])
def test_labels_follow_the_oracle(mvs_lib, oracle_lib, W, H, holes):
    import torch
    from paper_2104_06165_gb300 import scenes
    sc = scenes.make_scene(W=16, H=16, n_src=1, seed=1)
    known, depth, hyp, valid, cost = _inputs(W, H, holes, W + H)
    gw, gh = (W + 1) // 2, (H + 1) // 2
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        for iters in (1, 2):
            label = np.zeros((gh, gw), np.int32)
            mvs_lib.mvs_phi_mrf(ctx.h, known, depth, hyp, valid, cost, mvs_lib.PhiParams(trw_iters=iters), label)
            olabel, gap = oracle_lib.phi_mrf(known, depth.astype(np.float64), hyp.astype(np.float64), valid,
                                             cost.astype(np.float64), iters=iters)
            clear = gap > GAP
            assert np.array_equal(label < 0, olabel < 0) and np.array_equal(label == -2, olabel == -2)
            assert (label[clear] == olabel[clear]).all()
            assert clear.mean() > 0.9
