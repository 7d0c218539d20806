"""GPU parity of the GEMM that gathers filter windows itself (network stems, odd channel counts, small strided images)."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import TOL, run_conv, assert_conv_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
@pytest.mark.parametrize("C,K,R,stride,pad,H,W,resid", [
    (1, 8, 1, 1, 0, 1, 1, False),       # one element
    (3, 16, 3, 2, 1, 19, 23, False),    # a stem; one K block, its tail padding
    (3, 64, 7, 2, 3, 66, 70, True),     # 7 x 7 windows, more than one tile, ragged
    (5, 20, 3, 1, 0, 9, 9, True),       # no padding
    (37, 33, 5, 3, 4, 40, 17, False),   # windows far outside the image, output rows that are no 16-byte multiples
    (101, 129, 1, 1, 0, 13, 11, True),  # 1x1 with an odd channel count, two column tiles
    (4, 24, 11, 2, 5, 17, 17, False),   # the largest odd window the repack takes
    (64, 48, 3, 2, 1, 8, 8, True),      # four channels at a time, split K
    (20, 300, 3, 1, 1, 7, 9, False),    # four channels, any number of output channels
    (50, 256, 3, 1, 1, 12, 12, False),  # fp32 words one by one: the most output channels
])
def test_gathered_windows(C, K, R, stride, pad, H, W, resid, math):
    L = dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=stride, pad=pad, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    rng = np.random.default_rng([C, K, R, H])
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, R, R)) * np.sqrt(2.0 / (C * R * R))).astype(np.float32)
    b = rng.uniform(-1, 1, K).astype(np.float32)
    oh, ow = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - R) // stride + 1
    add = rng.uniform(-1, 1, (K, oh, ow)).astype(np.float32) if resid else None
    v = nb.VAR_GEMM1X1 if R == 1 else nb.VAR_IM2COL
    plan = nb.Plan([L], [0], [0])
    assert nb.nnv_exec_workspace_bytes(plan, 0, v, math) == 0      # no matrix of the windows in memory
    y = run_conv(plan, 0, L, v, math, x, w, b, add)
    assert_conv_close(y, omodel.run_layer(L, x, w, b, add), TOL[math])


@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
@pytest.mark.parametrize("C,K,R,stride,pad,H,W", [
    (3, 16, 3, 2, 1, 19, 23),           # gathered word by word
    (64, 48, 3, 2, 1, 8, 8),            # gathered four channels at a time
    (64, 40, 3, 1, 1, 7, 7),            # boxes of a small image
    (64, 64, 3, 1, 1, 40, 40),          # read in place by the TMA
    (333, 300, 1, 1, 0, 7, 7),          # explicit im2col (TF32)
])
def test_nan_pixels_stay_nan(C, K, R, stride, pad, H, W, math):
    """A NaN input -- with the bits the GPU's own arithmetic gives it, which integer rounding carries out of the exponent -- reaches
    exactly the outputs whose window holds it."""
    L = dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=stride, pad=pad, groups=1, H=H, W=W, in0=-1, in1=-1, act=0, has_bias=0)
    rng = np.random.default_rng([C, K, 5])
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    h, w0, c = H // 2, W // 2, C - 1
    x.view(np.uint32)[c, h, w0] = 0x7FFFFFFF
    w = (rng.standard_normal((K, C, R, R)) * np.sqrt(2.0 / (C * R * R))).astype(np.float32)
    y = run_conv(nb.Plan([L]), 0, L, nb.VAR_GEMM1X1 if R == 1 else nb.VAR_IM2COL, math, x, w)
    p, q = np.arange(y.shape[1]) * stride - pad, np.arange(y.shape[2]) * stride - pad
    hit = ((p <= h) & (h < p + R))[:, None] & ((q <= w0) & (w0 < q + R))[None, :]
    assert hit.any() and np.array_equal(np.isnan(y), np.broadcast_to(hit, y.shape))
