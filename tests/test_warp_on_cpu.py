"""The searches and rotations of csrc/peel.cuh with a CPU thread per lane (warp_on_cpu.cpp), against the oracle: nothing
keeps the lanes together but the barriers and votes that the source names."""
import os
import subprocess

import numpy as np
import pytest

import oracle

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2605_26845_b200", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("warp") / "warp_on_cpu")
    subprocess.run(["g++", "-std=c++20", "-O1", "-w", "-pthread", "-I", "/usr/local/cuda/include", "-I", CSRC,
                    os.path.join(HERE, "warp_on_cpu.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("N,pieces,k_max", [(3, 4, 9), (8, 14, 60), (17, 40, 30), (33, 60, 10), (64, 90, 8), (70, 40, 6), (230, 12, 3)])
def test_lanes_that_run_apart_find_the_same_schedule(program, N, pieces, k_max):
    rng = np.random.default_rng(N)
    A = np.zeros((N, N), np.int32)
    for _ in range(pieces):                              # balanced, so that nothing is padded
        A[np.arange(N), rng.permutation(N)] += rng.integers(1, 20)
    done = subprocess.run([program], input=np.array([N, k_max], np.int32).tobytes() + A.tobytes(), capture_output=True,
                          timeout=120, check=True)
    count = int(np.frombuffer(done.stdout[:4], np.int32)[0])
    ref = oracle.bvn_decompose(A[None], k_max)
    assert count == ref["count"][0]
    coef = np.frombuffer(done.stdout[4:4 + 4 * count], np.int32)
    perm = np.frombuffer(done.stdout[4 + 4 * count:], np.uint8).reshape(count, N)
    assert (coef == ref["coef"][0, :count]).all() and (perm == ref["perm"][0, :count]).all()
