"""GPU parity of the fp32 tile GEMM with fewer output channels a block and the input channels in four or eight parts: channels that end inside a part, a block
of 32 or a group of 16, every number of tiles that a form of the kernel takes."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import assert_conv_close, run_conv
from test_abi_wino_rule import rule

pytestmark = pytest.mark.gpu

# As for the kernel's other form: operands rounded to 2^-9 of a word cost 2.6e-2 / 4.9e-2 of the result through these transforms; fp32 words (2^-24) in the
# operands, the products' sums and both data transforms four times 2^-15 of that.
TOL = {nb.VAR_WINO_F4: 3.2e-6, nb.VAR_WINO_F6: 6.0e-6}


@pytest.mark.parametrize("variant,C,K,H,W,groups", [
    (nb.VAR_WINO_F4, 960, 16, 12, 16, 1),        # twelve tiles, whole parts
    (nb.VAR_WINO_F4, 300, 70, 11, 12, 1),        # nine; ten blocks of 32 in eight parts, the last one cut; outputs end inside a group
    (nb.VAR_WINO_F4, 1100, 33, 3, 3, 1),         # one
    (nb.VAR_WINO_F4, 1024, 250, 8, 12, 2),       # six; quarters
    (nb.VAR_WINO_F6, 130, 40, 12, 17, 2),        # six; five blocks in four parts
    (nb.VAR_WINO_F6, 330, 20, 23, 16, 1),        # twelve
    (nb.VAR_WINO_F6, 1030, 48, 6, 11, 1),        # two
])
def test_parts_of_the_input_channels(variant, C, K, H, W, groups):
    m = 4 if variant == nb.VAR_WINO_F4 else 6
    r = rule(m, C, K, -(-H // m) * -(-W // m))
    assert r["small"] and r["groups"] == groups
    L = dict(op=nb.OP_CONV, C=C, K=K, R=3, S=3, stride=1, pad=1, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    rng = np.random.default_rng([29, C, K, H, W])
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, 3, 3)) * np.sqrt(2.0 / (9 * C))).astype(np.float32)
    b = rng.uniform(-1, 1, K).astype(np.float32)
    add = rng.uniform(-1, 1, (K, H, W)).astype(np.float32)
    plan = nb.Plan([L])
    y = run_conv(plan, 0, L, variant, nb.MATH_TF32, x, w, b, add)
    assert_conv_close(y, omodel.run_layer(L, x, w, b, add), TOL[variant])
    assert np.array_equal(y, run_conv(plan, 0, L, variant, nb.MATH_TF32, x, w, b, add))
