"""GPU parity of the GEMM's write-out and loads where they can go wrong: column tiles that both groups of warps share or that leave one
idle, rows and columns that end inside a tile, K loops on both sides of where two more warps load operands, splits of every size."""
import numpy as np
import pytest

from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from gpu_util import TOL, assert_conv_close, run_conv

pytestmark = pytest.mark.gpu

SHAPES = [                  # C, K, H, W, residual
    (32, 20, 3, 11, True),       # one K block, 33 rows, 20 columns
    (160, 100, 9, 7, False),     # five K blocks: two loading warps
    (192, 36, 12, 8, True),      # six: four, three whole quarters of rows
    (232, 48, 43, 3, False),     # eight, the last one partly filled; 129 rows
    (300, 130, 5, 5, True),      # ten; columns end inside a 16-byte word, plain stores
]


@pytest.mark.parametrize("C,K,H,W,residual", SHAPES)
def test_every_column_tile_and_split(C, K, H, W, residual):
    rng = np.random.default_rng([3, C, K, H, W])
    x = rng.uniform(-1, 1, (C, H, W)).astype(np.float32)
    w = (rng.standard_normal((K, C, 1, 1)) * np.sqrt(2.0 / C)).astype(np.float32)
    b = rng.uniform(-1, 1, K).astype(np.float32)
    add = rng.uniform(-1, 1, (K, H, W)).astype(np.float32) if residual else None
    L = dict(op=nb.OP_CONV, C=C, K=K, R=1, S=1, stride=1, pad=0, groups=1, H=H, W=W, in0=-1, in1=-1, act=1, has_bias=1)
    ref = omodel.run_layer(L, x, w, b, add)
    for math in (nb.MATH_TF32, nb.MATH_BF16):
        for bn in (16, 32, 48, 64, 96, 128):
            for sp in (1, 2, 4, 8):
                if sp > -(-C // 32):
                    continue
                nb.nnv_tuning_set("gemm_tile=%d,%d" % (bn, sp))
                try:
                    y = run_conv(nb.Plan([L], [0], [0]), 0, L, nb.VAR_GEMM1X1, math, x, w, b, add)
                finally:
                    nb.nnv_tuning_set(None)
                assert_conv_close(y, ref, TOL[math], (nb.MATH_NAMES[math], bn, sp))
