"""GPU parity of the vectorised 3x3 depthwise kernel and of the pooling / layout kernels at the edges of their tiles."""
import numpy as np
import pytest
import torch

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import TOL, run_conv, assert_conv_close, chw_to_hwc, hwc_to_chw, dev, poisoned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,stride,pad,H,W", [
    (4, 1, 1, 1, 1),          # one quad, one pixel
    (132, 1, 1, 9, 7),        # 33 quads: two blocks of 17
    (128, 2, 1, 10, 10),      # a full block of 32 quads, one pixel per thread
    (96, 2, 1, 41, 39),       # two pixels per thread, ragged rows
    (32, 1, 0, 100, 97),      # four pixels per thread, no padding
])
def test_depthwise_tiles(C, stride, pad, H, W):
    L = dict(op=nb.OP_CONV, C=C, K=C, R=3, S=3, stride=stride, pad=pad, groups=C, H=H, W=W, in0=-1, in1=-1, act=2, has_bias=1)
    rng = np.random.default_rng(C + H)
    x = rng.uniform(-2, 2, (C, H, W)).astype(np.float32)
    w = rng.standard_normal((C, 1, 3, 3)).astype(np.float32)
    b = rng.uniform(-1, 1, C).astype(np.float32)
    oh, ow = (H + 2 * pad - 3) // stride + 1, (W + 2 * pad - 3) // stride + 1
    add = rng.uniform(-1, 1, (C, oh, ow)).astype(np.float32)
    plan = nb.Plan([L])
    y = run_conv(plan, 0, L, nb.VAR_DEPTHWISE, nb.MATH_FP32, x, w, b, add)
    assert_conv_close(y, omodel.run_layer(L, x, w, b, add), TOL[nb.MATH_FP32])


@pytest.mark.parametrize("C,R,stride,pad,H,W", [(4, 2, 2, 0, 4, 4), (36, 3, 2, 1, 7, 9), (64, 3, 1, 1, 5, 5)])
def test_maxpool_four_channels(C, R, stride, pad, H, W):
    L = dict(op=nb.OP_MAXPOOL, C=C, K=C, R=R, S=R, stride=stride, pad=pad, groups=1, H=H, W=W, in0=-1, in1=-1, act=0, has_bias=0)
    x = np.random.default_rng(C).uniform(-1, 1, (C, H, W)).astype(np.float32)
    oh, ow = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - R) // stride + 1
    d_out = poisoned(4 * oh * ow * C)
    nb.nnv_pool_exec(nb.Plan([L]), 0, dev(chw_to_hwc(x)), d_out, torch.cuda.current_stream())
    y = hwc_to_chw(d_out[:4 * oh * ow * C].view(torch.float32).reshape(oh, ow, C).cpu().numpy())
    assert np.array_equal(y, omodel.run_layer(L, x).astype(np.float32))


@pytest.mark.parametrize("C,H,W", [(1, 1, 1), (3, 8, 8), (3, 7, 5), (4, 31, 33), (5, 6, 7), (64, 7, 7), (33, 40, 1)])
def test_layout_conversions(C, H, W):
    x = np.random.default_rng(C * H).standard_normal((C, H, W)).astype(np.float32)
    d_hwc, d_chw = poisoned(4 * x.size), poisoned(4 * x.size)
    nb.nnv_chw_to_hwc(dev(x), d_hwc, C, H, W, torch.cuda.current_stream())
    nb.nnv_hwc_to_chw(d_hwc, d_chw, C, H, W, torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert np.array_equal(d_hwc[:4 * x.size].view(torch.float32).cpu().numpy().reshape(H, W, C), chw_to_hwc(x))
    assert np.array_equal(d_chw[:4 * x.size].view(torch.float32).cpu().numpy().reshape(C, H, W), x)
