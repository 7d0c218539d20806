"""GPU parity of the BF16 3x3 kernel where its rings are refilled and its write-out ends inside a tile: more channel blocks than box
slots, weight rings of every depth, output channels that are no multiple of four, patches that leave the image, with a residual."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import TOL, assert_conv_close, run_conv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,K,H,W", [
    (32, 30, 17, 9),        # one block; plain stores; a patch with one row and one with one column
    (160, 64, 20, 30),      # five blocks on four box slots
    (288, 100, 16, 8),      # nine blocks; columns end inside a chunk
    (544, 128, 9, 20),      # seventeen; wide tiles leave room for fewer weight boxes
])
def test_rings_and_edges(C, K, H, W):
    L = dict(op=nb.OP_CONV, C=C, K=K, R=3, S=3, stride=1, pad=1, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    rng = np.random.default_rng([13, C, K, H, W])
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, 3, 3)) * np.sqrt(2.0 / (9 * C))).astype(np.float32)
    b = rng.uniform(-1, 1, K).astype(np.float32)
    add = rng.uniform(-1, 1, (K, H, W)).astype(np.float32)
    ref = omodel.run_layer(L, x, w, b, add)
    for bn in (16, 48, 96, 128):
        for sp in (1, 2, 4, 8):
            if sp > C // 32:
                continue
            nb.nnv_tuning_set("conv3x3=1,%d,%d" % (bn, sp))
            try:
                y = run_conv(nb.Plan([L], [0], [0]), 0, L, nb.VAR_IM2COL, nb.MATH_BF16, x, w, b, add)
            finally:
                nb.nnv_tuning_set(None)
            assert_conv_close(y, ref, TOL[nb.MATH_BF16], (bn, sp))
