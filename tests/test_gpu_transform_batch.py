"""GPU parity of whole-model weight transformations that mix every kind of transform, at the edges of their blocks."""
import numpy as np
import pytest
import torch

from oracle import pack as opack
from oracle import winograd as owin
from paper_2206_07446_b200 import binding as nb
from gpu_util import dev, poisoned

pytestmark = pytest.mark.gpu

WINO_M = {nb.VAR_WINO_F2: 2, nb.VAR_WINO_F4: 4, nb.VAR_WINO_F6: 6}
MIX = [nb.VAR_IM2COL, nb.VAR_WINO_F6, nb.VAR_WINO_F2, nb.VAR_WINO_F4, nb.VAR_GEMM1X1]


# one padded filter block of 8; one block of 256 filters exactly, and one filter row more; several blocks and a remainder
@pytest.mark.parametrize("K,C", [(1, 1), (32, 8), (33, 8), (70, 64), (200, 72)])
def test_mixed_batch_matches_the_oracle(K, C):
    layers = [dict(op=nb.OP_CONV, C=C, K=K, R=1 if v == nb.VAR_GEMM1X1 else 3, S=1 if v == nb.VAR_GEMM1X1 else 3, stride=1,
                   pad=0 if v == nb.VAR_GEMM1X1 else 1, groups=1, H=8, W=8, in0=-1, in1=-1, act=0, has_bias=0) for v in MIX]
    rng = np.random.default_rng(K * C)
    ws = [rng.standard_normal((K, C, L["R"], L["S"])).astype(np.float32) for L in layers]
    w_off, pos = [], 0
    for w in ws:
        w_off.append(pos)
        pos += (w.nbytes + 255) // 256 * 256
    blob = np.zeros(pos, np.uint8)
    for w, o in zip(ws, w_off):
        blob[o:o + w.nbytes] = w.reshape(-1).view(np.uint8)
    plan = nb.Plan(layers, w_off, [0] * len(layers))
    ch = [(v, nb.MATH_TF32, 0) for v in MIX]
    offs, total = nb.nnv_transformed_layout(plan, ch)
    d_src, d_w = dev(blob), poisoned(pos)
    runs = []
    for _ in range(2):                                          # the batch reads what the stream wrote just before it
        out = poisoned(total)
        d_w.fill_(0xEE)
        d_w[:pos].copy_(d_src[:pos])
        nb.nnv_transform_all(plan, ch, d_w, pos, out, total, torch.cuda.current_stream())
        runs.append(out[:total].clone())                        # and what follows in the stream reads the results of all of it
    torch.cuda.synchronize()
    for i, v in enumerate(MIX):
        nbytes = nb.nnv_transformed_bytes(plan, i, v, nb.MATH_TF32)
        got = [r[offs[i]:offs[i] + nbytes].view(torch.float32).cpu().numpy() for r in runs]
        assert np.array_equal(got[0].view(np.uint32), got[1].view(np.uint32))
        if v in WINO_M:
            ref = owin.pad_channels(owin.filter_transform(ws[i], WINO_M[v]), -(-C // 8) * 8)
            assert np.max(np.abs(got[0].reshape(ref.shape) - ref)) / np.max(np.abs(ref)) <= 1e-5
        else:
            assert np.array_equal(got[0].view(np.uint32), opack.pack_weights(ws[i]).reshape(-1).view(np.uint32))
