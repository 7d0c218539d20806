"""GPU parity of Winograd layers that run as one launch from their raw weights: passes over small images, with the same bits in every way that a pass
gets its weights, and the layers on the other side of the rule beside them."""
import numpy as np
import pytest

import workloads as wl
from oracle import model as omodel
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness

pytestmark = pytest.mark.gpu

# Products of bf16 parts (layers of more tiles) lose 2^-16 of a word: rounded to 2^-9, operands cost 2.6e-2 / 4.9e-2 of the result through these
# transforms, so 2.0e-4 / 3.8e-4 a layer at most, and there are three.
TOL = {nb.VAR_WINO_F4: 6.0e-4, nb.VAR_WINO_F6: 1.2e-3}


def _model(C, K, H, W, pad, act, bias):
    """C -> K -> C -> C, the second layer's output added to the third's where it has the size."""
    oh, ow = H + 2 * pad - 2, W + 2 * pad - 2
    a = dict(op=nb.OP_CONV, C=C, K=K, R=3, S=3, stride=1, pad=pad, groups=1, H=H, W=W, in0=-1, in1=-1, act=act, has_bias=bias)
    c = dict(a, C=K, K=C, H=oh, W=ow, in0=0, act=0)
    d = dict(c, C=C, K=C, H=oh + 2 * pad - 2, W=ow + 2 * pad - 2, in0=1, in1=1 if pad == 1 else -1, act=act)
    layers = [a, c, d]
    ws, bs = wl.make_weights(layers, seed=31)
    return harness.model_from_workload(layers, ws, bs, wl.weight_blob), wl.make_input(layers, seed=31), layers, ws, bs


@pytest.mark.parametrize("variant,C,K,H,W,pad,act,bias", [
    (nb.VAR_WINO_F4, 512, 512, 7, 7, 1, 1, 1),         # eight slices of 64, two groups of tiles
    (nb.VAR_WINO_F4, 256, 256, 14, 14, 1, 2, 1),       # sixteen tiles: the tensor cores'
    (nb.VAR_WINO_F4, 128, 128, 10, 11, 1, 0, 1),       # nine tiles, five groups
    (nb.VAR_WINO_F4, 4, 3, 2, 3, 1, 0, 0),             # less than a tile, a slice, a block of outputs; the second layer's three channels are another kernel's
    (nb.VAR_WINO_F4, 36, 40, 5, 18, 1, 1, 1),          # channels and outputs that end inside their blocks
    (nb.VAR_WINO_F4, 64, 64, 23, 21, 1, 1, 1),         # more tiles still
    (nb.VAR_WINO_F4, 100, 132, 11, 8, 0, 2, 1),         # no padding
    (nb.VAR_WINO_F4, 72, 200, 6, 5, 2, 1, 0),          # an output larger than the input
    (nb.VAR_WINO_F4, 516, 64, 6, 6, 1, 1, 1),          # too many channels for it, then 64 -> 516
    (nb.VAR_WINO_F6, 512, 512, 5, 5, 1, 1, 1),         # one tile
    (nb.VAR_WINO_F6, 384, 512, 12, 10, 1, 0, 1),       # four tiles, two a block
    (nb.VAR_WINO_F6, 136, 64, 17, 14, 1, 1, 1),        # nine tiles
    (nb.VAR_WINO_F6, 128, 156, 4, 6, 1, 2, 0),
])
def test_small_image_layers(variant, C, K, H, W, pad, act, bias):
    m, x, layers, ws, bs = _model(C, K, H, W, pad, act, bias)
    want = np.asarray(omodel.run_model(layers, ws, bs, x)[-1], np.float64)
    ch = [(variant, nb.MATH_TF32, nb.ARM_RAW)] * 3
    zero_copy = [(variant, nb.MATH_TF32, nb.ARM_ZERO_COPY)] * 3
    runs = {"resident": m.resident_run(x, ch, depth=0)[0], "resident, staged": m.resident_run(x, ch, depth=2)[0], "cold": m.cold_run(x, ch, depth=0)[0],
            "cold, staged": m.cold_run(x, ch, depth=1)[0], "resident, zero-copy arm": m.resident_run(x, zero_copy, depth=0)[0]}
    runs = {name: np.array(y, np.float64).reshape(want.shape) for name, y in runs.items()}
    for name, y in runs.items():
        rel = np.linalg.norm(y - want) / np.linalg.norm(want)
        assert rel <= TOL[variant], (name, rel)
        assert np.array_equal(y, runs["resident"]), name
    # the stages timed each and the transformed weights of a warm run, through the kernels of prepared weights: the same bits
    timed = np.array(m.resident_run(x, ch, depth=0, want_timings=True)[0], np.float64).reshape(want.shape)
    assert np.array_equal(timed, runs["resident"])
    m.cold_run_continuous(x, ch, ch)
    assert np.array_equal(np.array(m.warm_run(x, ch)[0], np.float64).reshape(want.shape), runs["resident"])
