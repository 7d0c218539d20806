"""GPU parity of implicit GEMMs whose activation is small: tiles of whole image rows fetched as boxes, and the shapes next to
them that keep the explicit path; BF16 math also through the 3x3 halo kernel."""
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
    (24, 32, 3, 1, 20, 16),        # 320 pixels: tiles of 106 rows do not exist, explicit path
    (64, 64, 3, 0, 9, 9),          # no padding: explicit path
])
@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
def test_small_images(C, K, R, pad, H, W, math):
    L = dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=1, pad=pad, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    tol, err2, ref2 = TOL[math], 0.0, 0.0
    for seed in range(4):
        rng = np.random.default_rng([seed, C, K, H])
        x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
        w = (rng.standard_normal((K, C, R, R)) * np.sqrt(2.0 / (C * R * R))).astype(np.float32)
        b = rng.uniform(-0.1, 0.1, K).astype(np.float32)
        add = rng.uniform(-1, 1, (K, H + 2 * pad - R + 1, W + 2 * pad - R + 1)).astype(np.float32)
        ref = omodel.run_layer(L, x, w, b, add)
        y = run_conv(nb.Plan([L]), 0, L, nb.VAR_IM2COL, math, x, w, b, add)
        assert np.all(np.isfinite(y)) and np.max(np.abs(y - ref)) <= 8 * tol * np.max(np.abs(ref))
        err2 += float(np.sum((y - ref) ** 2))
        ref2 += float(np.sum(ref ** 2))
    assert np.sqrt(err2 / ref2) <= tol
