"""The search for the shape of a one-launch inverted-residual block: it is made once a plan, whatever a model's blocks are and however many passes plan
their launches, and not before the weights are on their way."""
import ctypes
import os

import numpy as np
import pytest

import workloads as wl
from workloads.configs import _Net
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness

pytestmark = pytest.mark.gpu


def searches():
    f = nb._lib.nnv_internal_ib_searches
    f.restype = ctypes.c_uint64
    return f()


def blocks_net(res, blocks):
    """A first convolution and inverted-residual blocks (expansion by 6) of the given (outputs, stride)."""
    n = _Net(3, res, res)
    x, cin = n.conv(-1, 32, 3, stride=2, act=wl.ACT_RELU6), 32
    for c, stride in blocks:
        h = n.conv(x, cin * 6, 1, pad=0, act=wl.ACT_RELU6)
        h = n.conv(h, cin * 6, 3, stride=stride, groups=cin * 6, act=wl.ACT_RELU6)
        x = n.conv(h, c, 1, pad=0, act=wl.ACT_NONE, add=x if stride == 1 and cin == c else -1)
        cin = c
    return n.layers


BLOCKS = [(32, 1), (32, 2), (64, 2), (64, 1), (96, 1), (96, 1), (160, 2), (160, 1)]


def _model(res, graphs):
    layers = blocks_net(res, BLOCKS)
    ws, bs = wl.make_weights(layers, seed=2)
    m = harness.model_from_workload(layers, ws, bs, wl.weight_blob, use_graphs=graphs)
    return m, wl.make_input(layers, seed=2)


@pytest.mark.parametrize("math", [nb.MATH_TF32, nb.MATH_BF16])
@pytest.mark.parametrize("res", [96, 160, 209, 210])
def test_a_plan_searches_once(res, math):
    m, x = _model(res, 0)
    ch = m.default_choices(prefer=[nb.VAR_GEMM1X1, nb.VAR_IM2COL], math=math)
    before = searches()
    y = m.cold_run(x, ch, depth=0)[0]
    first = searches()
    assert 0 < first - before <= len(BLOCKS)
    for _ in range(3):
        assert np.array_equal(m.cold_run(x, ch, depth=0)[0], y)
    assert searches() == first
    m.resident_run(x, ch, depth=0)                             # (the block whose weights are in two merged copies runs as one launch here)
    first = searches()
    assert first - before <= len(BLOCKS)
    m.resident_run(x, ch, depth=0)
    assert searches() == first


def test_not_before_the_weights_are_on_their_way(tmp_path):
    """A pass that fails at the first read of its weights has searched for nothing."""
    m, x = _model(96, 0)
    ch = m.default_choices(prefer=[nb.VAR_GEMM1X1, nb.VAR_IM2COL], math=nb.MATH_TF32)
    path = str(tmp_path / "m.nnv")
    m.write_model_file(path, ch)
    cache = nb.CacheFile(path)
    os.truncate(path, 8192)
    before = searches()
    with pytest.raises(nb.NnvError):
        m.cold_run_file(x, ch, cache, depth=0)
    assert searches() == before
