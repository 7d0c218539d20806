"""GPU: the F(4,3) and F(6,3) filter transforms are no further from the exact result than sums that take the middle tap's product, add the first
tap's and then the last one's, each multiply-add rounded once (with F(6,3) sums that begin with both outer taps are 5 % further off)."""
import numpy as np
import pytest
import torch

from oracle import winograd as owin
from paper_2206_07446_b200 import binding as nb
from gpu_util import dev, poisoned, rel_l2

pytestmark = pytest.mark.gpu


def _row(g, v):
    """g . v in single precision: a product of two words is exact in double precision, so each step rounds once."""
    s = (v[1].astype(np.float64) * g[1]).astype(np.float32)
    for k in (0, 2):
        s = (v[k].astype(np.float64) * g[k] + s).astype(np.float32)
    return s


@pytest.mark.parametrize("variant,m", [(nb.VAR_WINO_F4, 4), (nb.VAR_WINO_F6, 6)])
@pytest.mark.parametrize("C,K", [(64, 64), (40, 72), (256, 128)])
def test_no_further_from_exact_than_plain_multiply_adds(variant, m, C, K):
    w = (np.random.default_rng([m, C, K]).standard_normal((K, C, 3, 3)) * np.sqrt(2.0 / (9 * C))).astype(np.float32)
    exact = owin.filter_transform(w, m)                       # [a * a][K][C]
    G = owin.matrices(m)[1].astype(np.float32).astype(np.float64)
    a = m + 2
    plain = np.empty((a, a, K, C), np.float32)
    for nu in range(a):
        t = [_row(G[nu], [w[:, :, i, s] for s in range(3)]) for i in range(3)]
        for xi in range(a):
            plain[xi, nu] = _row(G[xi], t)
    L = dict(op=nb.OP_CONV, C=C, K=K, R=3, S=3, stride=1, pad=1, groups=1, H=14, W=14, in0=-1, in1=-1, act=1, has_bias=0)
    plan = nb.Plan([L])
    out = poisoned(nb.nnv_transformed_bytes(plan, 0, variant, nb.MATH_TF32))
    nb.nnv_transform_weights(plan, 0, variant, nb.MATH_TF32, dev(w), out, torch.cuda.current_stream())
    torch.cuda.synchronize()
    Cp = (C + 7) // 8 * 8
    got = out[:4 * a * a * K * Cp].view(torch.float32).reshape(a * a, K, Cp)[..., :C].cpu().numpy()
    assert rel_l2(got, exact) <= 1.01 * rel_l2(plain.reshape(a * a, K, C), exact)
