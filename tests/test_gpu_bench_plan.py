"""The benchmark times the plan a user has: inverted-residual blocks run as one launch in its headline steps, and it counts the kernels that it launched."""
import json
import os
import subprocess
import sys

import pytest

import workloads as wl
from oracle import selection as osel
from paper_2206_07446_b200 import binding as nb

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_headline_runs_what_a_plain_plan_runs(tmp_path):
    layers = wl.cfg3_mobilenetv2()
    costs = []
    for i, L in enumerate(layers):                              # a cost table that takes every 1x1 layer to the GEMM
        for v in osel.eligible(L):
            for m in osel.math_modes(v):
                best = v == (nb.VAR_GEMM1X1 if L["R"] == 1 else nb.VAR_DEPTHWISE if L["groups"] > 1 else nb.VAR_IM2COL) and m != nb.MATH_BF16
                costs.append(dict(layer=i, variant=v, math=m, h2d_raw_ns=1000, xform_ns=0, h2d_cached_ns=1000, exec_ns=1000 if best else 100000, zc_ns=0))
    table, report = str(tmp_path / "costs.json"), str(tmp_path / "report.json")
    json.dump(costs, open(table, "w"))
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--config", "cfg3_mobilenetv2", "--steps", "4", "--warmup", "3", "--minimal",
                          "--depth-steps", "0", "--no-cpu-baseline", "--also", "", "--load-costs", table, "--report", report],
                         cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    line = json.loads(out.stdout.strip().splitlines()[-1])
    rep = json.load(open(report))
    assert {c[0] for c in rep["breakdown"]["choices"] if c} == {"im2col", "gemm1x1", "depthwise"}
    # 52 layers, the layout conversions and the transforms; of the 16 blocks with an expansion most are one launch instead of three
    assert line["gpu_launches"] % 8 == 0 and 20 <= line["gpu_launches"] // 8 <= 54 - 2 * 12 + 8
    assert line["gpu_launches"] // 8 == rep["run"]["kernel_launches_per_step"]
