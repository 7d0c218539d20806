"""GPU parity of the fp32 tile GEMM that F(4,3) and F(6,3) layers of a few tiles run on: every number of tiles it takes, channels that end
inside its blocks of 32 and 64, and the layers on the other side of its rule."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import assert_conv_close, run_conv

pytestmark = pytest.mark.gpu

# Operands rounded to bf16 (2^-9 of a word) cost 2.6e-2 / 4.9e-2 of the result through these transforms; fp32 words (2^-24) in the operands, the
# products' sums and both data transforms four times 2^-15 of that: 3.2e-6 / 6.0e-6.
TOL = {nb.VAR_WINO_F4: 3.2e-6, nb.VAR_WINO_F6: 6.0e-6}


@pytest.mark.parametrize("variant,C,K,H,W", [
    (nb.VAR_WINO_F4, 64, 64, 3, 2),        # one tile, clipped
    (nb.VAR_WINO_F4, 512, 512, 7, 7),      # four
    (nb.VAR_WINO_F4, 40, 70, 5, 18),       # ten; channels end inside a block of 32, outputs inside one of 64
    (nb.VAR_WINO_F4, 8, 3, 8, 9),          # six; fewer channels than a block
    (nb.VAR_WINO_F4, 36, 200, 16, 5),      # eight
    (nb.VAR_WINO_F4, 33, 40, 9, 14),       # twelve, padded channels
    (nb.VAR_WINO_F6, 100, 130, 6, 6), (nb.VAR_WINO_F6, 256, 256, 11, 12), (nb.VAR_WINO_F6, 72, 64, 7, 19), (nb.VAR_WINO_F6, 64, 96, 17, 18),
])
def test_few_tiles(variant, C, K, H, W):
    L = dict(op=nb.OP_CONV, C=C, K=K, R=3, S=3, stride=1, pad=1, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    rng = np.random.default_rng([23, C, K, H, W])
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, 3, 3)) * np.sqrt(2.0 / (9 * C))).astype(np.float32)
    b = rng.uniform(-1, 1, K).astype(np.float32)
    add = rng.uniform(-1, 1, (K, H, W)).astype(np.float32)
    y = run_conv(nb.Plan([L], [0], [0]), 0, L, variant, nb.MATH_TF32, x, w, b, add)
    err = assert_conv_close(y, omodel.run_layer(L, x, w, b, add), TOL[variant])
    print("rel %.2e" % err)
    assert np.array_equal(y, run_conv(nb.Plan([L], [0], [0]), 0, L, variant, nb.MATH_TF32, x, w, b, add))
