"""One-launch inverted-residual blocks in every kind of pass that weights can come to them in: each layer's output has the bits that a run with timings, which
launches the layers one by one, gives it, whether the weights come in one copy, in several, through staging slots, from a model file, through preparation queues
or prepared by an earlier pass."""
import ctypes

import numpy as np
import pytest

import workloads as wl
from workloads.configs import _Net
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness

pytestmark = pytest.mark.gpu


def launches():
    f = nb._lib.nnv_internal_ib_launches
    f.restype = ctypes.c_uint64
    return f()


def _net():
    """Three blocks in a row with biases, two of them with a residual, behind a 1x1 layer and in front of another."""
    n = _Net(8, 23, 19)
    x, cin = n.conv(-1, 32, 1, pad=0, act=wl.ACT_RELU6, bias=1), 32
    for c, stride in ((32, 1), (64, 2), (64, 1)):
        h = n.conv(x, cin * 6, 1, pad=0, act=wl.ACT_RELU6, bias=1)
        h = n.conv(h, cin * 6, 3, stride=stride, groups=cin * 6, act=wl.ACT_RELU6, bias=1)
        x = n.conv(h, c, 1, pad=0, act=wl.ACT_NONE, add=x if stride == 1 and cin == c else -1, bias=1)
        cin = c
    n.conv(x, 96, 1, pad=0, act=wl.ACT_RELU6, bias=1)
    return n.layers


def _model(graphs):
    layers = _net()
    ws, bs = wl.make_weights(layers, seed=8)
    bs = [b + np.linspace(-0.5, 0.5, b.size, dtype=np.float32) for b in bs]            # (biases away from zero)
    return harness.model_from_workload(layers, ws, bs, wl.weight_blob, max_depth=8, use_graphs=graphs), wl.make_input(layers, seed=8)


@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
def test_every_layer_has_its_bits(math, graphs, tmp_path):
    m, x = _model(graphs)
    n = len(m.layers)
    ch = [(nb.VAR_DEPTHWISE, nb.MATH_FP32, 0) if L["groups"] > 1 else (nb.VAR_GEMM1X1, math, 0) for L in m.layers]
    zc = [(c[0], c[1], nb.ARM_ZERO_COPY if c[0] == nb.VAR_GEMM1X1 else nb.ARM_RAW) for c in ch]
    m.resident_run(x, ch, depth=0, want_timings=True)
    want = [m.layer_output(i) for i in range(n)]
    assert all(np.all(np.isfinite(w)) for w in want)

    def check(name, run, times=2, fused=True):
        before = launches()
        for rep in range(times):
            if m.arena is not None:
                m.arena.fill_(0xFF)
            y = run()[0]
            assert np.array_equal(y.reshape(want[-1].shape).view(np.uint32), want[-1].view(np.uint32)), (name, rep)
            for i in range(n):
                got = m.layer_output(i)
                assert np.array_equal(got.view(np.uint32), want[i].view(np.uint32)), (name, rep, i, int((got != want[i]).sum()))
        assert (launches() > before) == fused, name

    m.ensure_arena(ch, 0)
    check("resident", lambda: m.resident_run(x, ch, depth=0))
    for depth in (4, 6, 8):
        check("resident, %d slots" % depth, lambda: m.resident_run(x, ch, depth=depth))
    check("cold", lambda: m.cold_run(x, ch, depth=0))
    check("cold, zero-copy arm", lambda: m.cold_run(x, zc, depth=0), fused=False)      # (the depthwise weights are copied, in copies of their own)
    for depth in (6, 8) if not graphs else (4, 5, 6):
        check("cold, %d slots" % depth, lambda: m.cold_run(x, ch, depth=depth))
    path = str(tmp_path / "blocks.nnv")
    m.write_model_file(path, ch)
    cache = nb.CacheFile(path)
    for depth in (0, 6):
        check("file, %d slots" % depth, lambda: m.cold_run_file(x, ch, cache, depth=depth))
    for queues, queue_of in ((2, [1 + i % 2 for i in range(n)]), (3, [i % 4 for i in range(n)]), (2, [0] * n)):      # (0: the execution stream)
        check("queues", lambda: m.cold_run_queues(x, ch, queue_of, queues))
    m.d_warm = harness.dev_bytes(nb.nnv_warm_bytes(m.plan, ch, m.w_bytes))              # (poisoned)
    check("continuous", lambda: m.cold_run_continuous(x, ch, ch), times=1)
    check("warm", lambda: m.warm_run(x, ch), times=3)
    direct = [(nb.VAR_DEPTHWISE, nb.MATH_FP32, 0) if L["groups"] > 1 else (nb.VAR_DIRECT, nb.MATH_FP32, 0) for L in m.layers]
    m.d_warm.fill_(0xFF)
    m.cold_run_continuous(x, direct, ch)                        # the warm kernels' weights are prepared behind the cold inference
    check("warm after another cold choice", lambda: m.warm_run(x, ch), times=3)
    nb.nnv_tuning_set("merge=0")
    try:
        check("cold, a copy a layer", lambda: m.cold_run(x, ch, depth=0))
        for spec in ("chunk=16,16", "chunk=64,256"):            # blocks whose weights are in two copies run apart
            nb.nnv_tuning_set(spec)
            before = launches()
            for _ in range(2):
                y = m.cold_run(x, ch, depth=0)[0]
                assert np.array_equal(y.reshape(want[-1].shape).view(np.uint32), want[-1].view(np.uint32)), spec
            assert launches() - before < (1 if graphs else 2) * 3, spec
    finally:
        nb.nnv_tuning_set(None)
    assert nb.nnv_device_status() == 0
