"""Every form of the one-launch Winograd layer -- tiles a block, slices of the input channels, tiles and channels that end inside a block -- against the oracle and,
bit for bit, against the kernels for transformed weights."""
import ctypes

import numpy as np
import pytest

import workloads as wl
from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness
from gpu_util import assert_conv_close
from test_abi_wino_rule import rule

pytestmark = pytest.mark.gpu

# Operands rounded to 2^-9 of a word cost 2.6e-2 / 4.9e-2 of the result through these transforms; fp32 words (2^-24) in the operands, the products' sums
# and both data transforms four times 2^-15 of that.
TOL = {nb.VAR_WINO_F4: 3.2e-6, nb.VAR_WINO_F6: 6.0e-6}


@pytest.mark.parametrize("variant,C,K,H,W,T,slices", [
    (nb.VAR_WINO_F4, 4, 3, 11, 13, 2, 4),        # twelve tiles of one quad
    (nb.VAR_WINO_F4, 64, 70, 11, 12, 2, 4),      # nine: the last block has one
    (nb.VAR_WINO_F4, 256, 250, 3, 15, 2, 4),     # four
    (nb.VAR_WINO_F4, 260, 64, 6, 8, 2, 8),       # channels that end inside a block of 32
    (nb.VAR_WINO_F4, 512, 500, 4, 12, 2, 8),     # three
    (nb.VAR_WINO_F6, 12, 16, 17, 24, 1, 4),      # twelve
    (nb.VAR_WINO_F6, 64, 33, 12, 23, 1, 4),      # eight
    (nb.VAR_WINO_F6, 192, 500, 6, 5, 1, 4),      # one
    (nb.VAR_WINO_F6, 260, 64, 5, 18, 1, 8),      # three
    (nb.VAR_WINO_F6, 100, 700, 12, 11, 2, 4),    # two tiles a block
    (nb.VAR_WINO_F6, 300, 500, 6, 17, 2, 8),     # the last block has one
])
def test_forms(variant, C, K, H, W, T, slices):
    m = 4 if variant == nb.VAR_WINO_F4 else 6
    r = rule(m, C, K, -(-H // m) * -(-W // m))
    assert r["layer"] and (r["T"], r["slices"]) == (T, slices)
    L = dict(op=nb.OP_CONV, C=C, K=K, R=3, S=3, stride=1, pad=1, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    ws, bs = wl.make_weights([L], seed=33)
    x = wl.make_input([L], seed=33)
    model = harness.model_from_workload([L], ws, bs, wl.weight_blob)
    ch = [(variant, nb.MATH_TF32, nb.ARM_RAW)]
    y = model.resident_run(x, ch, depth=0)[0].reshape(K, H, W).copy()
    assert_conv_close(y, omodel.run_layer(L, x[0], ws[0], bs[0], None), TOL[variant])
    own = model.resident_run(x, ch, depth=0, want_timings=True)[0].reshape(K, H, W)
    assert np.array_equal(y, own)
    assert nb.nnv_device_status() == 0


@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
def test_block_of_more_than_256_outputs(math):
    """An inverted-residual block whose projection's weights come in two boxes, in both maths."""
    def conv(C, K, R, in0, groups=1, act=0):
        return dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=1, pad=R // 2, groups=groups, H=10, W=10, in0=in0, in1=-1, act=act, has_bias=1)
    layers = [conv(8, 64, 1, -1, act=1), conv(64, 256, 1, 0, act=2), conv(256, 256, 3, 1, 256, act=1), conv(256, 288, 1, 2)]
    ws, bs = wl.make_weights(layers, seed=34)
    x = wl.make_input(layers, seed=34)
    m = harness.model_from_workload(layers, ws, bs, wl.weight_blob)
    ch = [(nb.VAR_DEPTHWISE, nb.MATH_FP32, 0) if L["groups"] > 1 else (nb.VAR_GEMM1X1, math, 0) for L in layers]
    m.resident_run(x, ch, depth=0, want_timings=True)
    want = [m.layer_output(i) for i in range(4)]
    counter = nb._lib.nnv_internal_ib_launches
    counter.restype = ctypes.c_uint64
    before = counter()
    m.resident_run(x, ch, depth=0)
    assert counter() == before + 1
    for i in range(4):
        assert np.array_equal(m.layer_output(i).view(np.uint32), want[i].view(np.uint32)), i
