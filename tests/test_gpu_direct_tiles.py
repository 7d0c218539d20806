"""GPU parity of the direct kernel on larger tiles: both tile sizes, every split over a cluster, and the edges of its chunks and groups."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import TOL, run_conv, assert_conv_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,K,R,stride,pad,H,W", [
    (64, 128, 3, 2, 1, 57, 55),          # 64 x 64 tiles over clusters of eight, ragged rows
    (512, 512, 3, 1, 1, 7, 7),           # 32 x 32 over eight
    (200, 477, 3, 2, 1, 10, 10),         # an odd number of quads, K no multiple of four
    (88, 36, 3, 1, 1, 9, 7),             # less than a tile of either
    (16, 48, 3, 1, 1, 33, 33),           # 32 x 32 over two
    (64, 64, 3, 1, 1, 113, 111),         # several waves
    (256, 256, 3, 2, 0, 29, 30),         # no padding
    (128, 96, 3, 1, 2, 14, 14),          # more padding than the filter needs
    (24, 884, 1, 2, 0, 141, 142),        # 1x1: fewer quads than a chunk, 64 x 64 unsplit
    (1024, 256, 1, 1, 0, 14, 14), (2048, 512, 1, 1, 0, 7, 7), (68, 130, 1, 1, 0, 60, 61), (960, 162, 1, 1, 0, 7, 7), (2048, 1000, 1, 1, 0, 1, 1),
])
def test_tiles(C, K, R, stride, pad, H, W):
    L = dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=stride, pad=pad, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    rng = np.random.default_rng(C * K + H)
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, R, R)) * np.sqrt(2.0 / (C * R * R))).astype(np.float32)
    b = rng.uniform(-0.1, 0.1, K).astype(np.float32)
    oh, ow = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - R) // stride + 1
    add = rng.uniform(-1, 1, (K, oh, ow)).astype(np.float32)
    plan = nb.Plan([L])
    y = run_conv(plan, 0, L, nb.VAR_DIRECT, nb.MATH_FP32, x, w, b, add)
    assert_conv_close(y, omodel.run_layer(L, x, w, b, add), TOL[nb.MATH_FP32])
    assert np.array_equal(y, run_conv(plan, 0, L, nb.VAR_DIRECT, nb.MATH_FP32, x, w, b, add))
