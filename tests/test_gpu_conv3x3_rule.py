"""GPU parity of 3x3 TF32 layers on both sides of the rule that picks the halo kernel or the implicit GEMM."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import TOL, run_conv, assert_conv_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,K,H,W", [
    (32, 100, 150, 141),      # 128-column GEMM tiles that do not fit the GPU at once: halo kernel, ragged channels and edges
    (32, 48, 150, 141),       # the same image where they do
    (384, 130, 48, 62),       # twelve channel blocks on 48 patches: halo kernel, K split
    (384, 128, 48, 56),       # 21 patches: implicit GEMM
])
def test_both_sides_of_the_rule(C, K, H, W):
    L = dict(op=nb.OP_CONV, C=C, K=K, R=3, S=3, stride=1, pad=1, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    rng = np.random.default_rng(C + K)
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, 3, 3)) * np.sqrt(2.0 / (9 * C))).astype(np.float32)
    b = rng.uniform(-1, 1, K).astype(np.float32)
    y = run_conv(nb.Plan([L], [0], [0]), 0, L, nb.VAR_IM2COL, nb.MATH_TF32, x, w, b)
    assert_conv_close(y, omodel.run_layer(L, x, w, b), TOL[nb.MATH_TF32])
