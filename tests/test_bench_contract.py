"""The benchmark's reference arm (the CPU oracle on a bounded sample) prints one JSON line
with the keys the benchmark contract names; what is computed of the counters, and the count of launches."""
import json
import os
import re
import subprocess
import sys

import numpy as np
import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_the_contract_line():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--config", "2",
                          "--steps", "1", "--warmup", "0"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert out.returncode == 0, out.stderr
    lines = [l for l in out.stdout.splitlines() if l.strip()]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["unit"] == "decompositions/s" and d["higher_is_better"] is True
    assert d["value"] > 0 and d["steps"] == 1 and d["n_gpus"] == 1 and d["vs_baseline"] is None
    assert d["dtype"] == "int32" and d["data"] == "synthetic" and "workload" in d["config"]
    cb = d["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["cores"] >= 1 and cb["value"] == d["value"] and cb["sample"]
    assert d["e2e"] == {"value": d["value"], "unit": d["unit"], "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}


def test_other_ranks_of_the_reference_arm_do_nothing():
    env = dict(os.environ, RANK="1", WORLD_SIZE="2", LOCAL_RANK="1")
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--gpus", "2"],
                         capture_output=True, text=True, timeout=120, cwd=ROOT, env=env)
    assert out.returncode == 0 and out.stdout.strip() == ""


def test_operations_are_those_of_the_kernel_that_is_timed():
    """Few ranks are decomposed without searches, so what the searching kernel counts is not set against that kernel's time."""
    work = np.ones((3, 10))
    few, more = bench.operations(work, work, bench.FEW_RANKS), bench.operations(work, work, bench.FEW_RANKS + 1)
    assert few["bvn_decompose"] is None and few["mw_decompose"] is not None and more["bvn_decompose"] is not None
    assert bench.rate_of(None, 1.0) == (None, None) and bench.over(None, 2.0) is None
    assert bench.rate_of((3e6, 6e6), 1.0) == (3.0, 6.0) and bench.over(3.0, 2.0) == 1.5
    with open(os.path.join(ROOT, "paper_2605_26845_b200", "csrc", "small.cuh")) as f:
        assert int(re.search(r"SMALL_MAX_N = (\d+)", f.read()).group(1)) == bench.FEW_RANKS


@pytest.mark.gpu
@pytest.mark.parametrize("N,B,launches", [(8, 3, 4), (64, 100, 4), (64, 1300, 7)])
def test_launches_are_counted_in_a_capture(N, B, launches):
    """Greedy, Birkhoff and two scorings; in a batch too large for 32-bit entries the first and the last two launch twice."""
    import torch

    import paper_2605_26845_b200 as ms
    d = torch.ones((B, N, N), dtype=torch.int32, device="cuda")
    path = ms.Path(B, N, 2, 2)
    path.run(d)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        path.run(d)
    assert bench.kernels_in(graph.raw_cuda_graph()) == launches
