"""GPU parity of the fp32 direct kernel at the edges of its tiles, chunks and reduction splits."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import TOL, run_conv, assert_conv_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,K,R,S,stride,pad,H,W", [
    (8, 32, 3, 3, 1, 1, 8, 8),           # one chunk, exact tiles
    (12, 33, 3, 3, 1, 1, 7, 5),          # half a chunk of channels, ragged tiles, K not a multiple of 4
    (64, 128, 3, 3, 2, 1, 57, 55),       # 32 x 32 tiles
    (512, 36, 3, 3, 1, 1, 7, 7),         # 64 chunks over a cluster of eight
    (64, 64, 3, 3, 1, 1, 151, 149),      # 703 x 2 tiles, the last ones ragged
    (4, 5, 1, 1, 1, 0, 1, 1),            # a single output pixel
    (68, 40, 1, 1, 2, 0, 15, 13),        # 1x1, one channel word beyond a chunk
    (256, 512, 1, 1, 1, 0, 14, 14),
    (32, 130, 1, 1, 1, 0, 100, 99),
    (3, 64, 7, 7, 2, 3, 40, 37),         # flat reduction: stem
    (5, 7, 3, 3, 1, 0, 9, 11),           # flat reduction: odd channels, no padding
    (8, 16, 5, 3, 1, 2, 12, 12),         # flat reduction: other windows
])
def test_direct_shapes(C, K, R, S, stride, pad, H, W):
    L = dict(op=nb.OP_CONV, C=C, K=K, R=R, S=S, stride=stride, pad=pad, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    rng = np.random.default_rng(C * K + H)
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, R, S)) * np.sqrt(2.0 / (C * R * S))).astype(np.float32)
    b = rng.uniform(-0.1, 0.1, K).astype(np.float32)
    oh, ow = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - S) // stride + 1
    add = rng.uniform(-1, 1, (K, oh, ow)).astype(np.float32)
    plan = nb.Plan([L])
    y = run_conv(plan, 0, L, nb.VAR_DIRECT, nb.MATH_FP32, x, w, b, add)
    assert_conv_close(y, omodel.run_layer(L, x, w, b, add), TOL[nb.MATH_FP32])
    assert np.array_equal(y, run_conv(plan, 0, L, nb.VAR_DIRECT, nb.MATH_FP32, x, w, b, add))
