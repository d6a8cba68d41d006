"""Weight gradients and the fused backward passes at the sizes where their
kernels change: one-pixel levels, levels narrower than a 16-pixel step,
segments of 64 pixels cut by the border, odd level heights.  Each is compared
with the oracle on the library's own stored tensors: fp32 sums within the
bound of the layer-by-layer comparison, bf16 passes bit for bit."""
import numpy as np
import pytest

from oracle import cnn_oracle as cn
from test_gpu_cnn_layers import DEC, D_HI, D_LO, ENC, _check_f32, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W, H", [(16, 16), (80, 48), (208, 16), (144, 112)])
def test_gradients_at_ragged_sizes(mvs_lib, W, H):
    import torch
    m = mvs_lib
    rng = np.random.default_rng(W + H)
    img, plane, cost = _state(rng, W, H)
    _, target, _ = _state(rng, W, H)
    mask = (rng.uniform(size=(H, W)) < 0.7).astype(np.uint8)
    net = m.mvs_cnn_create(W, H, D_LO, D_HI, 31, torch.cuda.current_stream())
    try:
        theta = m.mvs_cnn_get_params(net).astype(np.float64)
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (img, plane, cost, target, mask)]
        m.mvs_cnn_backward(net, *dev)
        rd = lambda t, lv=0: m.mvs_cnn_read(net, t, lv, W, H).astype(np.float64)
        grads = cn.unpack(m.mvs_cnn_get_grads(net).astype(np.float64))
        weights = cn.unpack(theta)
        e = [rd(m.MVS_CNN_T_ENC, lv) for lv in range(5)]
        ge = [rd(m.MVS_CNN_T_GRAD_ENC, lv) for lv in range(5)]
        d = [rd(m.MVS_CNN_T_DEC, lv) for lv in range(4)]
        gd = [rd(m.MVS_CNN_T_GRAD_DEC, lv) for lv in range(4)]
        cat = [rd(m.MVS_CNN_T_CAT, lv) for lv in range(4)]
        gc = [rd(m.MVS_CNN_T_GRAD_CAT, lv) for lv in range(4)]
        gp = [rd(m.MVS_CNN_T_GRAD_POOL, lv) for lv in range(4)]
        pool = [rd(m.MVS_CNN_T_POOL, lv) for lv in range(4)]
        up_ch = [cn.LAYERS[DEC[lv]][0] - cn.LAYERS[ENC[lv]][1] for lv in range(4)]
        for lv in range(4):
            below, act = (gd[lv + 1], d[lv + 1]) if lv < 3 else (ge[4], e[4])
            assert np.array_equal(below, cn.to_bf16(cn.up_backward(gc[lv][..., :up_ch[lv]])) * (act > 0))
            expect = cn.to_bf16(gc[lv][..., up_ch[lv]:] + cn.pool_backward(gp[lv])) * (e[lv] > 0)
            assert np.array_equal(ge[lv], expect)
        assert not gd[0][d[0] <= 0].any()
        gouts, ins = {9: rd(m.MVS_CNN_T_GRAD_HEAD)}, {9: d[0]}
        for lv in range(4):
            gouts[DEC[lv]], ins[DEC[lv]] = gd[lv], cat[lv]
        for lv in range(5):
            gouts[ENC[lv]], ins[ENC[lv]] = ge[lv], rd(m.MVS_CNN_T_INPUT) if lv == 0 else pool[lv - 1]
        for li in range(10):
            w = weights[li][0]
            _, gw, gb = cn.conv_backward(ins[li], w, gouts[li])
            _, gwa, gba = cn.conv_backward(np.abs(ins[li]), w, np.abs(gouts[li]))
            h, wd = ins[li].shape[:2]
            # the tensor-core steps of a 64-pixel segment over the block's rows
            # (up to 16 dependent additions each), then one addition per block
            chain = 64 * h + -(-wd // 64) * h
            _check_f32(f"grad w {li}", grads[li][0], gw, gwa, chain)
            _check_f32(f"grad b {li}", grads[li][1], gb, gba, chain)
    finally:
        m.mvs_cnn_destroy(net)
