"""Which kernels the GPU tests of the direct tiles, of the one-launch blocks and of few-tile Winograd layers run (host arithmetic, no GPU): every path gives
results within the same tolerance, many the same bits, so those tests alone would not see a rule that has stopped choosing the kernel they are for."""
import ctypes

import pytest

from paper_2206_07446_b200 import binding as nb
from test_abi_wino_rule import rule


def direct(P, C, K, taps):
    out = (ctypes.c_int32 * 2)()
    nb._lib.nnv_internal_direct_rule(P, C, K, taps, out)
    return tuple(out)


@pytest.mark.parametrize("C,K,R,stride,pad,H,W,tile,splits", [
    (64, 128, 3, 2, 1, 57, 55, 64, 8), (512, 512, 3, 1, 1, 7, 7, 32, 8), (200, 477, 3, 2, 1, 10, 10, 32, 8), (88, 36, 3, 1, 1, 9, 7, 32, 8),
    (16, 48, 3, 1, 1, 33, 33, 32, 1), (64, 64, 3, 1, 1, 113, 111, 64, 1), (256, 256, 3, 2, 0, 29, 30, 32, 4), (128, 96, 3, 1, 2, 14, 14, 32, 8),
    (24, 884, 1, 2, 0, 141, 142, 64, 1), (1024, 256, 1, 1, 0, 14, 14, 32, 4), (2048, 512, 1, 1, 0, 7, 7, 32, 8), (68, 130, 1, 1, 0, 60, 61, 32, 1),
    (960, 162, 1, 1, 0, 7, 7, 32, 8), (2048, 1000, 1, 1, 0, 1, 1, 32, 8)])
def test_direct_tiles(C, K, R, stride, pad, H, W, tile, splits):
    P = ((H + 2 * pad - R) // stride + 1) * ((W + 2 * pad - R) // stride + 1)
    assert direct(P, C, K, R * R) == (tile, splits)


def block(bf16, C, E, K, H, W, stride, residual):
    out = (ctypes.c_int32 * 56)()
    return None if nb._lib.nnv_internal_ib_shape(bf16, C, E, K, H, W, stride, residual, out) else out[7]


@pytest.mark.parametrize("C,E,K,stride,H,W,residual,tf32,bf16", [      # CTAs that share a patch; None: three launches
    (16, 96, 24, 2, 112, 112, 0, 1, 1), (24, 144, 24, 1, 56, 56, 1, 2, 1), (24, 144, 32, 2, 57, 55, 0, 2, 4), (32, 192, 32, 1, 28, 28, 1, 2, 4),
    (64, 384, 64, 1, 14, 14, 1, 8, 8), (96, 576, 96, 1, 14, 13, 1, 16, 16), (96, 576, 160, 2, 15, 14, 0, 8, 16), (160, 960, 160, 1, 7, 7, 1, 16, None),
    (160, 960, 320, 1, 7, 7, 0, 16, None), (160, 960, 320, 1, 5, 9, 0, 16, None), (8, 48, 20, 1, 9, 33, 0, 2, 1), (256, 1024, 252, 2, 3, 2, 0, 16, None),
    (40, 120, 40, 1, 1, 1, 1, 2, 4), (64, 256, 288, 1, 10, 10, 0, 8, 8)])
def test_blocks(C, E, K, stride, H, W, residual, tf32, bf16):
    assert block(0, C, E, K, H, W, stride, residual) == tf32
    assert block(1, C, E, K, H, W, stride, residual) == bf16


@pytest.mark.parametrize("m,C,K,H,W,pad,small,layer", [                # of the three layers C -> K -> C -> C of the test: fp32 tile GEMM, one launch
    (4, 512, 512, 7, 7, 1, (1, 1, 1), (1, 1, 1)), (4, 256, 256, 14, 14, 1, (0, 0, 0), (0, 0, 0)), (4, 128, 128, 10, 11, 1, (1, 1, 1), (0, 0, 0)),
    (4, 4, 3, 2, 3, 1, (1, 1, 1), (0, 0, 0)), (4, 36, 40, 5, 18, 1, (1, 1, 1), (1, 1, 1)), (4, 64, 64, 23, 21, 1, (0, 0, 0), (0, 0, 0)),
    (4, 100, 132, 11, 8, 0, (1, 1, 1), (1, 0, 1)), (4, 72, 200, 6, 5, 2, (1, 1, 1), (1, 1, 1)), (4, 516, 64, 6, 6, 1, (1, 1, 1), (0, 1, 0)),
    (6, 512, 512, 5, 5, 1, (0, 0, 0), (0, 0, 0)), (6, 384, 512, 12, 10, 1, (0, 0, 1), (0, 0, 1)), (6, 136, 64, 17, 14, 1, (1, 1, 1), (0, 0, 0)),
    (6, 128, 156, 4, 6, 1, (1, 1, 1), (1, 0, 1))])
def test_winograd_layers(m, C, K, H, W, pad, small, layer):
    nb.nnv_tuning_set(None)
    h, w, got = H, W, []
    for c, k in ((C, K), (K, C), (C, C)):
        h, w = h + 2 * pad - 2, w + 2 * pad - 2
        got.append(rule(m, c, k, -(-h // m) * -(-w // m)))
    assert tuple(r["small"] for r in got) == small and tuple(r["layer"] for r in got) == layer
