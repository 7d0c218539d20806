"""Where inverted-residual blocks run as one launch: not where that would hold up the preparation of the next block, and with the same bits either way."""
import ctypes

import numpy as np
import pytest

import workloads as wl
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness
from test_gpu_block_search import blocks_net

pytestmark = pytest.mark.gpu

BLOCKS = [(32, 1), (64, 2), (64, 1), (96, 1)]


def launches():
    f = nb._lib.nnv_internal_ib_launches
    f.restype = ctypes.c_uint64
    return f()


def test_staging_and_queues():
    layers = blocks_net(96, BLOCKS)
    ws, bs = wl.make_weights(layers, seed=2)
    m = harness.model_from_workload(layers, ws, bs, wl.weight_blob, max_depth=8, use_graphs=0)
    x = wl.make_input(layers, seed=2)
    ch = m.default_choices(prefer=[nb.VAR_GEMM1X1, nb.VAR_IM2COL], math=nb.MATH_TF32)
    want = m.resident_run(x, ch, depth=0, want_timings=True)[0]

    def fused(run):
        before = launches()
        assert np.array_equal(run()[0], want)
        return launches() - before

    for depth, n in ((0, 4), (1, 0), (2, 0), (3, 0), (4, 4), (6, 4), (8, 4)):
        assert fused(lambda: m.resident_run(x, ch, depth=depth)) == n, depth
    for depth, n in ((1, 0), (3, 0), (4, 0), (5, 0), (6, 4), (8, 4)):
        assert fused(lambda: m.cold_run(x, ch, depth=depth)) == n, depth
    assert fused(lambda: m.cold_run(x, ch, depth=0)) == 3             # (the last layer's copy is not merged with the others')
    for queues, n in ((1, 0), (2, 4), (3, 4)):
        assert fused(lambda: m.cold_run_queues(x, ch, [1 + i % queues for i in range(len(layers))], queues)) == n, queues
    assert fused(lambda: m.cold_run_continuous(x, ch, ch)) == 4
    assert fused(lambda: m.warm_run(x, ch)) == 4
    m.plan = m.second_plan(use_graphs=1)                       # (its passes count the launches while they are recorded)
    for depth, n in ((3, 0), (4, 4)):
        assert fused(lambda: m.cold_run(x, ch, depth=depth)) == n, depth
        assert fused(lambda: m.cold_run(x, ch, depth=depth)) == 0, depth
    nb.nnv_tuning_set("block=0")
    try:
        assert fused(lambda: m.resident_run(x, ch, depth=0)) == 0
    finally:
        nb.nnv_tuning_set(None)
    assert nb.nnv_device_status() == 0
