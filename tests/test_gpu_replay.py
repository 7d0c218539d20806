"""Calls that replay a recorded pass without planning it: what no longer fits is refused as before, other arguments run another pass, and the
layers' outputs are those of the pass that ran last."""
import numpy as np
import pytest
import torch

import workloads as wl
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness

pytestmark = pytest.mark.gpu


def _model():
    layers = wl.tiny_net()
    ws, bs = wl.make_weights(layers, seed=5)
    return harness.model_from_workload(layers, ws, bs, wl.weight_blob), wl.make_input(layers, seed=5)


def _choices(m, prefer, math):
    return m.default_choices(prefer=prefer, math=math)


def test_resident_and_cold():
    m, x = _model()
    gemm, direct = _choices(m, [nb.VAR_GEMM1X1, nb.VAR_IM2COL], nb.MATH_TF32), _choices(m, [nb.VAR_DIRECT], nb.MATH_FP32)
    want = {}
    for name, ch in (("gemm", gemm), ("direct", direct)):
        want[name] = m.resident_run(x, ch, depth=0, want_timings=True)[0].copy(), [m.layer_output(i) for i in range(len(m.layers))]
    for rep in range(3):                                       # recorded, replayed, in turn
        for name, ch in (("gemm", gemm), ("direct", direct)):
            y = m.resident_run(x, ch, depth=0)[0]
            assert np.array_equal(y, want[name][0]), (rep, name)
            for i in range(len(m.layers)):
                assert np.array_equal(m.layer_output(i), want[name][1][i]), (rep, name, i)
    need = nb.nnv_arena_bytes(m.plan, gemm, 0)
    args = [m.plan, nb.choices_array(m.plan, gemm), m.d_weights, m.w_bytes, None, 0, m.d_input, m.d_output, m.arena, m.arena.numel(), m.streams[1], m.streams[2], 0]
    nb.nnv_resident_run(*args)
    for at, bad in ((9, need - 1), (3, 4), (12, 99), (4 + 4, m.arena[128:])):
        wrong = list(args)
        wrong[at] = bad
        with pytest.raises(nb.NnvError):
            nb.nnv_resident_run(*wrong)
    with pytest.raises(nb.NnvError):                           # the streams have to be two
        nb.nnv_resident_run(*args[:10], m.streams[2], m.streams[2], 0)
    y0 = m.cold_run(x, gemm, depth=0)[0]
    for _ in range(2):
        assert np.array_equal(m.cold_run(x, gemm, depth=0)[0], y0)
    args = [m.plan, nb.choices_array(m.plan, gemm), m.h_weights, m.w_bytes, None, 0, m.h_input, m.h_output, m.arena, need, *m.streams[:3], 0]
    nb.nnv_cold_run(*args)
    with pytest.raises(nb.NnvError):
        nb.nnv_cold_run(*args[:9], need - 1, *args[10:])
    unpinned = torch.zeros_like(m.h_output)                    # pageable memory: copied, not written in place
    nb.nnv_cold_run(*args[:7], unpinned, *args[8:])
    assert np.array_equal(unpinned.numpy(), y0)


def test_warm():
    m, x = _model()
    ch = _choices(m, [nb.VAR_GEMM1X1, nb.VAR_IM2COL], nb.MATH_TF32)
    y0 = m.cold_run_continuous(x, ch, ch)[0]
    for _ in range(3):
        assert np.array_equal(m.warm_run(x, ch)[0], y0)
    x2 = x[..., ::-1].copy()
    y2 = m.warm_run(x2, ch)[0]
    assert not np.array_equal(y2, y0) and np.array_equal(m.warm_run(None, ch)[0], y2)
    args = [m.plan, nb.choices_array(m.plan, ch), m.d_warm, m.warm_bytes, m.w_bytes, m.h_input, m.h_output, m.arena, m.arena.numel(), m.streams[1], m.streams[2]]
    nb.nnv_warm_run(*args)
    for at, bad in ((3, m.warm_bytes - 1), (8, nb.nnv_arena_bytes(m.plan, ch, 0) // 2), (4, 4)):
        wrong = list(args)
        wrong[at] = bad
        with pytest.raises(nb.NnvError):
            nb.nnv_warm_run(*wrong)
    m.h_input.copy_(torch.from_numpy(np.ascontiguousarray(x)).reshape(m.h_input.shape))
    nb.nnv_warm_run(*args)
    assert np.array_equal(m.h_output.numpy(), y0)
