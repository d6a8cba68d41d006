"""Message passing over more strips of eight node rows than blocks fit on the
device, so that blocks walk a second and a third strip with the rings, buffers
and polls of the one before, against the FP64 oracle."""
import numpy as np
import pytest

from test_gpu_trw import GAP, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W, H", [(36, 2500), (2, 4900), (150, 2600), (34, 7400)])
@pytest.mark.parametrize("holes", [0.05, 0.5, 1.0])
def test_labels_follow_the_oracle(mvs_lib, oracle_lib, W, H, holes):
    import torch
    from paper_2104_06165_gb300 import scenes
    # a block per multiprocessor at most: more strips than that
    assert -(-H // 2) > 8 * torch.cuda.get_device_properties(0).multi_processor_count
    sc = scenes.make_scene(W=16, H=16, n_src=1, seed=1)
    known, depth, hyp, valid, cost = _inputs(W, H, holes, W + H)
    label = np.zeros(((H + 1) // 2, (W + 1) // 2), np.int32)
    with mvs_lib.Context(sc.K, sc.R, sc.t, sc.images, stream=torch.cuda.current_stream()) as ctx:
        for iters in (1, 2):
            mvs_lib.mvs_phi_mrf(ctx.h, known, depth, hyp, valid, cost, mvs_lib.PhiParams(trw_iters=iters), label)
            olabel, gap = oracle_lib.phi_mrf(known, depth.astype(np.float64), hyp.astype(np.float64), valid,
                                             cost.astype(np.float64), iters=iters)
            clear = gap > GAP
            assert np.array_equal(label < 0, olabel < 0) and np.array_equal(label == -2, olabel == -2)
            assert (label[clear] == olabel[clear]).all()
            assert clear.mean() > 0.9
