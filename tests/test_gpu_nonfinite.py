"""Infinities and NaN through the kernels of few-tile Winograd layers, whole layers from raw weights, larger direct tiles and one-launch inverted-residual
blocks: outputs that the value reaches are what the plain sum gives, all others are as if it was not there."""
import numpy as np
import pytest

import workloads as wl
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness
from gpu_util import run_conv

pytestmark = pytest.mark.gpu

VALUES = [np.inf, -np.inf, np.nan]


def _case(C, K, R, H, W, seed):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, R, R)) * np.sqrt(2.0 / (C * R * R))).astype(np.float32)
    return x, w


def _layer(C, K, R, H, W, stride=1, act=0, in0=-1, in1=-1, groups=1):
    return dict(op=nb.OP_CONV, C=C, K=K, R=R, S=R, stride=stride, pad=R // 2, groups=groups, H=H, W=W, in0=in0, in1=in1, act=act, has_bias=0)


@pytest.mark.parametrize("value", VALUES)
@pytest.mark.parametrize("C,K,R,stride,H,W", [(64, 96, 3, 1, 21, 19), (200, 100, 3, 2, 10, 11), (512, 70, 1, 1, 9, 7), (16, 48, 3, 1, 33, 33)])
def test_direct(C, K, R, stride, H, W, value):
    x, w = _case(C, K, R, H, W, 5)
    L = _layer(C, K, R, H, W, stride)
    plan = nb.Plan([L])
    clean = run_conv(plan, 0, L, nb.VAR_DIRECT, nb.MATH_FP32, x, w)
    c, h, v = C - 3, H // 2, W - 2
    bad = x.copy()
    bad[c, h, v] = value
    y = run_conv(plan, 0, L, nb.VAR_DIRECT, nb.MATH_FP32, bad, w)
    want = clean.copy()
    for r in range(R):
        for s in range(R):
            oh, ow = h + L["pad"] - r, v + L["pad"] - s
            if oh % stride == 0 and ow % stride == 0 and 0 <= oh // stride < y.shape[1] and 0 <= ow // stride < y.shape[2]:
                want[:, oh // stride, ow // stride] = value * w[:, c, r, s]
    assert np.array_equal(np.isnan(y), np.isnan(want))
    assert np.array_equal(y[~np.isnan(want)], want[~np.isnan(want)])


@pytest.mark.parametrize("value", VALUES)
@pytest.mark.parametrize("variant,C,K,H,W", [(nb.VAR_WINO_F4, 64, 70, 8, 8), (nb.VAR_WINO_F4, 36, 40, 11, 12), (nb.VAR_WINO_F4, 512, 64, 7, 7),
                                             (nb.VAR_WINO_F4, 960, 16, 12, 16), (nb.VAR_WINO_F6, 100, 64, 12, 12), (nb.VAR_WINO_F6, 40, 33, 17, 18)])
def test_few_tiles(variant, C, K, H, W, value):
    """The transforms carry a value to all of its tiles' outputs (as infinities of both signs: NaN); other tiles do not change."""
    m = 4 if variant == nb.VAR_WINO_F4 else 6
    x, w = _case(C, K, 3, H, W, 6)
    L = _layer(C, K, 3, H, W)
    bad = x.copy()
    c, h, v = C - 1, m if H > 2 * m else 1, m if W > 2 * m else 1           # (in two tiles a row and column, or in one)
    bad[c, h, v] = value
    touched = np.zeros((H, W), bool)
    for th in range(-(-H // m)):
        for tw in range(-(-W // m)):
            if th * m - 1 <= h < th * m + m + 1 and tw * m - 1 <= v < tw * m + m + 1:
                touched[th * m:th * m + m, tw * m:tw * m + m] = True
    assert touched.any() and not touched.all()
    plan = nb.Plan([L])
    outs = [(run_conv(plan, 0, L, variant, nb.MATH_TF32, x, w), run_conv(plan, 0, L, variant, nb.MATH_TF32, bad, w))]
    if C <= 512:                                                # the whole layer from raw weights
        mod = harness.model_from_workload([L], [w], [None], wl.weight_blob)
        ch = [(variant, nb.MATH_TF32, nb.ARM_RAW)]
        clean = mod.resident_run(x[None], ch, depth=0)[0].reshape(K, H, W).copy()
        outs.append((clean, mod.resident_run(bad[None], ch, depth=0)[0].reshape(K, H, W).copy()))
    for clean, y in outs:
        assert np.all(np.isfinite(clean))
        assert np.array_equal(y[:, ~touched], clean[:, ~touched])
        assert not np.any(np.isfinite(y[:, h, v]))
        assert np.all(~np.isfinite(y[:, touched]) | (y[:, touched] == clean[:, touched]))


@pytest.mark.parametrize("value", VALUES)
@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
@pytest.mark.parametrize("where", ["input", "expansion", "depthwise", "projection"])
def test_blocks(where, math, value):
    """Every layer of a block as the three launches give it, whichever operand holds the value."""
    C, E, K, H, W = 32, 192, 32, 15, 13
    layers = [_layer(C, C, 1, H, W, act=0), _layer(C, E, 1, H, W, act=2, in0=0), _layer(E, E, 3, H, W, act=1, in0=1, groups=E),
              _layer(E, K, 1, H, W, in0=2, in1=0)]
    ws, bs = wl.make_weights(layers, seed=4)
    x = wl.make_input(layers, seed=4)
    if where == "input":
        x[0, 5, 7, 6] = value
    else:
        w = ws[("expansion", "depthwise", "projection").index(where) + 1]
        w.reshape(-1)[w.size // 2 + 3] = value
    ch = [(nb.VAR_DEPTHWISE, nb.MATH_FP32, 0) if L["groups"] > 1 else (nb.VAR_GEMM1X1, math, 0) for L in layers]
    m = harness.model_from_workload(layers, ws, bs, wl.weight_blob)
    m.resident_run(x, ch, depth=0, want_timings=True)
    want = [m.layer_output(i) for i in range(4)]
    m.resident_run(x, ch, depth=0)
    for i in range(4):
        got = m.layer_output(i)
        assert np.array_equal(np.isnan(got), np.isnan(want[i])), i
        assert np.array_equal(got[~np.isnan(got)], want[i][~np.isnan(got)]), i
