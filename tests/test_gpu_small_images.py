"""GPU parity of im2col GEMMs whose activation is small: tiles of whole image rows fetched as boxes and rounded by the kernel, and the
shapes next to them, which are gathered; BF16 math also through the 3x3 halo kernel."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import TOL, run_conv, assert_conv_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,K,R,pad,H,W", [
    (64, 40, 3, 1, 7, 7),          # one tile of 49 rows
    (32, 64, 3, 1, 14, 14),        # two tiles of seven image rows
    (36, 33, 3, 1, 5, 9),          # C not a multiple of 32, odd K
    (96, 48, 5, 2, 8, 6),          # 5x5
    (64, 64, 3, 1, 1, 1),          # one pixel
    (24, 32, 3, 1, 20, 16),        # 320 pixels: no equal tiles of whole rows
    (64, 64, 3, 0, 9, 9),          # no padding: the output is not the image's size
])
@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
def test_small_images(C, K, R, pad, H, W, math):
    L = dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=1, pad=pad, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    for seed in range(4):
        rng = np.random.default_rng([seed, C, K, H])
        x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
        w = (rng.standard_normal((K, C, R, R)) * np.sqrt(2.0 / (C * R * R))).astype(np.float32)
        b = rng.uniform(-0.1, 0.1, K).astype(np.float32)
        add = rng.uniform(-1, 1, (K, H + 2 * pad - R + 1, W + 2 * pad - R + 1)).astype(np.float32)
        ref = omodel.run_layer(L, x, w, b, add)
        y = run_conv(nb.Plan([L]), 0, L, nb.VAR_IM2COL, math, x, w, b, add)
        assert_conv_close(y, ref, TOL[math], seed)


@pytest.mark.parametrize("C,K,R,H,W", [(64, 64, 3, 14, 14), (164, 40, 3, 14, 14), (96, 48, 5, 8, 6), (64, 128, 3, 7, 7), (64, 64, 1, 9, 5)])
def test_small_tf32_activations_are_rounded(C, K, R, H, W):
    """Both operands rounded to nearest: errors uniform in +-2^-11 of the value's power of two, rms 2.8e-4 of it and 1.9e-4 of the
    value, for two operands 2.7e-4.  An activation truncated by the tensor core has twice that error itself, in all 4.2e-4."""
    L = dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=1, pad=R // 2, groups=1, H=H, W=W, in0=-1, in1=-1, act=0, has_bias=0)
    for seed in range(4):
        rng = np.random.default_rng([seed, C, K, H, 1])
        x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
        w = (rng.standard_normal((K, C, R, R)) * np.sqrt(2.0 / (C * R * R))).astype(np.float32)
        y = run_conv(nb.Plan([L]), 0, L, nb.VAR_IM2COL, nb.MATH_TF32, x, w)
        assert_conv_close(y, omodel.run_layer(L, x, w, None, None), 3.4e-4, seed)


@pytest.mark.parametrize("tuning", ["gemm_tile=16,1;gemm_ring=2", "gemm_tile=48,1;gemm_ring=3", "gemm_tile=32,1", "gemm_tile=32,2;gemm_ring=5",
                                    "gemm_tile=48,16", "gemm_tile=16,8;gemm_ring=2"])
def test_rounded_boxes_in_rings_that_wrap(tuning):
    """75 K blocks in rings of every kind, by one CTA or a cluster: two groups of warps round them in turn."""
    C, K, R, H, W = 96, 48, 5, 14, 14
    L = dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=1, pad=2, groups=1, H=H, W=W, in0=-1, in1=-1, act=2, has_bias=1)
    rng = np.random.default_rng(3)
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, R, R)) * np.sqrt(2.0 / (C * R * R))).astype(np.float32)
    b, add = rng.uniform(-0.1, 0.1, K).astype(np.float32), rng.uniform(-1, 1, (K, H, W)).astype(np.float32)
    nb.nnv_tuning_set(tuning)
    try:
        y = run_conv(nb.Plan([L]), 0, L, nb.VAR_IM2COL, nb.MATH_TF32, x, w, b, add)
    finally:
        nb.nnv_tuning_set(None)
    assert_conv_close(y, omodel.run_layer(L, x, w, b, add), 3.4e-4, tuning)
