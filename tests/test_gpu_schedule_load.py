"""Algorithm 1 on a model whose executions are short beside its reads: preparations do not move to the execution queue, where the other queues' copies go
first, because they look free there."""
import statistics
import time

import numpy as np
import pytest
import torch

import workloads as wl
from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200 import harness

pytestmark = pytest.mark.gpu


def test_resnet50_schedule_is_no_slower_than_reads_in_turn():
    layers = wl.cfg4_resnet50()
    ws, bs = wl.make_weights(layers)
    x = wl.make_input(layers)
    m = harness.model_from_workload(layers, ws, bs, wl.weight_blob, use_graphs=0)
    costs = nb.CostTable([c for c in m.profile(x, reps=5) if c["math"] != nb.MATH_BF16])
    ch, queue_of, _, _ = m.schedule(x, costs, 2, allow_cached=0, rounds=2, eps_pct=1, combo_limit=4096)
    need, streams = m.ensure_arena(ch, 0), m.prep_streams(2)

    def ms(queues):
        ts = []
        for _ in range(12):
            torch.cuda.synchronize()
            t = time.perf_counter()
            nb.nnv_cold_run_queues(m.plan, ch, queues, 2, m.h_weights, m.w_bytes, None, 0, m.h_input, m.h_output, m.arena, need, streams, False)
            ts.append(1e3 * (time.perf_counter() - t))
        return statistics.median(ts[2:]), m.h_output.numpy().copy()

    (found, y), (in_turn, z) = ms(queue_of), ms([1 + i % 2 for i in range(len(layers))])
    assert np.array_equal(y, z)
    assert found <= 1.12 * in_turn, (found, in_turn, queue_of)
