"""GPU parity of the one-launch inverted-residual block: every layer's output has the bits that the three layers' own launches
give it (a run with per-operation timings launches them one by one), at the edges of its patches and channel blocks."""
import numpy as np
import pytest

import workloads as wl
from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness
from gpu_util import rel_l2

pytestmark = pytest.mark.gpu


def _conv(C, K, R, H, W, in0, stride=1, groups=1, in1=-1, act=0, bias=0):
    return dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=stride, pad=R // 2, groups=groups, H=H, W=W, in0=in0, in1=in1, act=act, has_bias=bias)


# C, E, K, stride, H, W, bias, residual: one and several channel blocks, ragged ones, one CTA a patch, accumulators and whole splits a
# CTA, more than 256 output channels, patches cut by the image's edge, odd and one-pixel grids
SHAPES = [(16, 96, 24, 2, 112, 112, 0, 0), (24, 144, 24, 1, 56, 56, 0, 1), (24, 144, 32, 2, 57, 55, 1, 0), (32, 192, 32, 1, 28, 28, 1, 1),
          (64, 384, 64, 1, 14, 14, 0, 1), (96, 576, 96, 1, 14, 13, 1, 1), (96, 576, 160, 2, 15, 14, 0, 0), (160, 960, 160, 1, 7, 7, 1, 1),
          (160, 960, 320, 1, 7, 7, 0, 0), (160, 960, 320, 1, 5, 9, 1, 0), (8, 48, 20, 1, 9, 33, 1, 0), (256, 1024, 252, 2, 3, 2, 1, 0), (40, 120, 40, 1, 1, 1, 1, 1)]


@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
@pytest.mark.parametrize("shape", SHAPES)
def test_block_has_the_bits_of_its_layers(shape, math):
    C, E, K, stride, H, W, bias, residual = shape
    oh, ow = (H - 1) // stride + 1, (W - 1) // stride + 1
    layers = [_conv(C, C, 1, H, W, -1, act=1, bias=bias), _conv(C, E, 1, H, W, 0, act=2, bias=bias),
              _conv(E, E, 3, H, W, 1, stride, E, act=1, bias=bias)]
    if residual:
        assert K == C and stride == 1
    layers.append(_conv(E, K, 1, oh, ow, 2, in1=0 if residual else -1, bias=bias))
    ws, bs = wl.make_weights(layers, seed=3)
    bs = [None if b is None else b + np.linspace(-0.5, 0.5, b.size, dtype=np.float32) for b in bs]      # (biases away from zero)
    x = wl.make_input(layers, seed=3)
    model = harness.model_from_workload(layers, ws, bs, wl.weight_blob)
    ch = [(nb.VAR_DEPTHWISE, nb.MATH_FP32, 0) if L["groups"] > 1 else (nb.VAR_GEMM1X1, math, 0) for L in layers]
    y0, _ = model.resident_run(x, ch, depth=0, want_timings=True)
    own = [model.layer_output(i) for i in range(4)]
    acts = omodel.run_model(layers, ws, bs, x)
    tol = 3e-3 if math == nb.MATH_TF32 else 3e-2                # a chain of two GEMMs behind one: three times a GEMM's own
    for depth in (0, 3):
        y1, _ = model.resident_run(x, ch, depth=depth)
        for i in range(1, 4):
            got = model.layer_output(i)
            assert rel_l2(got, acts[i]) <= tol, (depth, i)
            assert np.array_equal(got.view(np.uint32), own[i].view(np.uint32)), (depth, i, int((got != own[i]).sum()), got.size)
        assert np.array_equal(y0.view(np.uint32), y1.view(np.uint32)), depth
    assert nb.nnv_device_status() == 0
