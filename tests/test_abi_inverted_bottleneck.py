"""The launch shape of the one-launch inverted-residual block (host arithmetic, no GPU): every place a CTA reads or writes in shared
memory lies where the layout says, and the CTAs of a cluster hold the projection's channel blocks in the order its own launch adds them."""
import ctypes
import os

import pytest

from paper_2206_07446_b200 import binding as nb

CSRC = os.path.join(os.path.dirname(os.path.abspath(nb.__file__)), "csrc")
NAMES = ("ph pw hw rows px tiles_h tiles_w ranks both step nb_most bn2 issuers tmem w1 conv d w2 bar par smem pairs").split()
PITCH, BARS = 144, 8 * 24


def up(v, a):
    return -(-v // a) * a


def shape(bf16, C, E, K, H, W, stride, residual):
    out = (ctypes.c_int32 * 56)()
    if nb._lib.nnv_internal_ib_shape(bf16, C, E, K, H, W, stride, residual, out):
        return None
    s = dict(zip(NAMES, out))
    s["blocks"] = [(out[24 + 2 * r], out[25 + 2 * r]) for r in range(s["ranks"])]
    return s


def gemm(bf16, M, N, nkb, addend):
    out = (ctypes.c_int32 * 13)()
    assert nb._lib.nnv_internal_gemm_shape(3 if bf16 else 0, M, N, 1, nkb, 1, addend, out) == 0
    return dict(splits=out[1], issuers=out[4])


@pytest.mark.parametrize("bf16", [0, 1])
def test_layout_and_order(bf16):
    seen = 0
    for C, E, K in [(8, 48, 20), (16, 96, 24), (24, 144, 24), (24, 144, 32), (32, 192, 64), (40, 120, 40), (64, 384, 64), (96, 576, 160),
                    (160, 960, 160), (160, 960, 320), (256, 1024, 252), (256, 512, 512), (32, 2048, 128)]:
        for H, W in [(1, 1), (3, 2), (5, 5), (7, 7), (9, 33), (14, 14), (28, 27), (57, 55), (112, 112)]:
            for stride in (1, 2):
                residual = int(C == K and stride == 1)
                s = shape(bf16, C, E, K, H, W, stride, residual)
                if s is None:
                    continue
                seen += 1
                oh, ow, nkb1, nkb2 = (H - 1) // stride + 1, (W - 1) // stride + 1, -(-C // 32), -(-E // 32)
                what = (bf16, C, E, K, H, W, stride, s)
                assert s["rows"] == s["hw"] * ((s["ph"] - 1) * stride + 3) <= 128 and s["hw"] == (s["pw"] - 1) * stride + 3, what
                assert s["px"] == s["ph"] * s["pw"] and s["tiles_h"] * s["ph"] >= oh and s["tiles_w"] * s["pw"] >= ow, what
                assert (s["tiles_h"] - 1) * s["ph"] < oh and (s["tiles_w"] - 1) * s["pw"] < ow, what
                # operands, then the expansion, then the received rows from 0 on; behind them the projection's operands, then its rows
                pad = lambda n: up(n, 8)
                xs, ds = up(s["rows"] * 128, 1024), pad(s["px"]) * 64 if bf16 else up(s["px"] * 128, 1024)
                w1, w2 = nkb1 * s["nb_most"] * (2048 if bf16 else 4096), s["nb_most"] * s["bn2"] * (64 if bf16 else 128)
                conv = nkb1 * pad(s["rows"]) * 64 if bf16 else 0
                rows_per = -(-s["px"] // s["ranks"])
                assert nkb1 * xs <= s["w1"] and s["w1"] + w1 <= s["conv"] and s["conv"] + conv <= s["d"], what
                assert s["nb_most"] * s["rows"] * PITCH <= s["d"], what
                assert s["ranks"] == 1 or s["ranks"] * rows_per * s["bn2"] * 4 <= s["d"], what
                assert s["d"] + s["nb_most"] * ds <= s["w2"] and s["w2"] + w2 <= s["bar"] and s["d"] + s["px"] * s["bn2"] * 4 <= s["bar"], what
                assert s["w1"] % 1024 == s["conv"] % 1024 == s["d"] % 1024 == s["w2"] % 1024 == s["par"] % 16 == s["bar"] % 8 == 0, what
                assert s["bar"] + BARS <= s["par"] + 8 and 1024 + s["par"] + 4 * (s["nb_most"] * 352 + s["bn2"]) <= s["smem"] <= 226 * 1024, what
                # an MMA reads 128 rows of A
                last = [(nkb1 - 1) * xs + 16384] if not bf16 else [s["conv"] + (nkb1 - 1) * pad(s["rows"]) * 64 + 3 * pad(s["rows"]) * 16 + 2048]
                last.append(s["d"] + (s["nb_most"] - 1) * ds + (16384 if not bf16 else 3 * pad(s["px"]) * 16 + 2048))
                assert 1024 + max(last) <= s["smem"], what
                # accumulators, and a cluster's CTA has an SM's shared memory as it has its TMEM columns
                assert s["tmem"] >= max(s["issuers"] * s["nb_most"] * 32, (1 + s["both"]) * s["bn2"]) and s["tmem"] in (32, 64, 128, 256, 512), what
                assert s["ranks"] == 1 or s["smem"] >= min(226 * 1024, 228 * 1024 * s["tmem"] // 512 - 1024), what
                assert s["bn2"] >= K and s["bn2"] % 16 == 0 and s["bn2"] <= (256 if s["both"] else 512) and s["nb_most"] <= 8, what
                # the K blocks of every accumulator, in the order the projection's own launch adds them
                g = gemm(bf16, oh * ow, K, nkb2, residual)
                e = gemm(bf16, H * W, E, nkb1, 0)
                assert e["splits"] == 1 and e["issuers"] == g["issuers"] == s["issuers"], what
                want = []
                for sp in range(g["splits"]):
                    k = list(range(nkb2 * sp // g["splits"], nkb2 * (sp + 1) // g["splits"]))
                    want.append([k] if s["step"] == 1 else [b for b in (k[0::2], k[1::2]) if b])
                got = [list(range(f, f + n * s["step"], s["step"])) for f, n in s["blocks"]]
                assert got == [b for split in want for b in split], what
                assert s["pairs"] == sum(1 << i for i, split in enumerate(want) if len(split) == 2), what
                assert s["both"] == (s["issuers"] == 2 and s["step"] == 1), what
    assert seen > 60


def test_the_next_kernel_is_let_in_after_the_tmem_allocation():
    body = open(os.path.join(CSRC, "inverted_bottleneck.cuh")).read().split("__global__")[1]
    assert body.index("tmem_take(") < body.index("pdl_wait();") < body.index("pdl_trigger();")
