"""The searches and rotations of csrc/peel.cuh and the bitmaps of csrc/small.cuh with a CPU thread per lane (warp_on_cpu.cpp),
against the oracle: nothing keeps the lanes together but the barriers and votes that the source names."""
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


def decompose(program, A, k_max, *how):
    N = A.shape[0]
    done = subprocess.run([program, *how], input=np.array([N, k_max], np.int32).tobytes() + A.tobytes(), capture_output=True,
                          timeout=120, check=True)
    count = int(np.frombuffer(done.stdout[:4], np.int32)[0])
    return (count, np.frombuffer(done.stdout[4:4 + 4 * count], np.int32),
            np.frombuffer(done.stdout[4 + 4 * count:], np.uint8).reshape(count, N))


@pytest.mark.parametrize("N,pieces,k_max", [(100, 30, 3), (128, 16, 3), (140, 12, 2), (170, 10, 2), (200, 8, 2)])
def test_every_number_of_words(program, N, pieces, k_max):
    """Four to seven words: the first level apart, chances counted or not, rows read back from entries of another layout."""
    rng = np.random.default_rng(N)
    A = np.zeros((N, N), np.int32)
    for _ in range(pieces):
        A[np.arange(N), rng.permutation(N)] += rng.integers(1, 20)
    count, coef, perm = decompose(program, A, k_max)
    ref = oracle.bvn_decompose(A[None], k_max)
    assert count == ref["count"][0]
    assert (coef == ref["coef"][0, :count]).all() and (perm == ref["perm"][0, :count]).all()


@pytest.mark.parametrize("N", range(1, 9))
@pytest.mark.parametrize("dense", [False, True])
def test_bitmaps_of_few_ranks(program, N, dense):
    rng = np.random.default_rng(10 * N + dense)
    for _ in range(2):
        A = np.zeros((N, N), np.int32)
        for _ in range(30 if dense else N):
            A[np.arange(N), rng.permutation(N)] += rng.integers(1, 4 if dense else 200)
        k_max = N * N + 1
        count, coef, perm = decompose(program, A, k_max, "small")
        ref = oracle.bvn_decompose(A[None], k_max)
        assert count == ref["count"][0]
        assert (coef == ref["coef"][0, :count]).all() and (perm == ref["perm"][0, :count]).all()


def smallest_matching(edges, column_of):
    """The lexicographically smallest perfect matching: row by row the lowest column that can be had without touching the rows
    before, by a search for a way to hand the row's own column on."""
    N = len(column_of)
    col, row = list(column_of), [0] * N
    for i, c in enumerate(col):
        row[c] = i
    for i in range(N):
        came = {col[i]: None}                            # columns that can be freed by giving col[i] away: who takes it from whom
        queue = [col[i]]
        for c in queue:
            for r in np.flatnonzero(edges[:, c]):
                if r > i and col[r] not in came:
                    came[col[r]] = c                     # row r can take c and frees its own
                    queue.append(col[r])
        mover, c, moves = i, min(c for c in came if edges[i, c]), []
        while True:
            moves.append((mover, c))
            if came[c] is None:
                break
            mover, c = row[c], came[c]
        for r, c in moves:
            col[r], row[c] = c, r
    return col


@pytest.mark.parametrize("N", [1, 2, 3, 8, 32, 64, 70, 100, 140, 170, 200, 230])
@pytest.mark.parametrize("kind", ["matching only", "tree", "cycles"])
def test_smallest_matching_of_an_adopted_graph(program, N, kind):
    """What the greedy decomposition does with its tight edges: rows on no cycle leave the graph before the searches. A matching
    and nothing else, hardly more than a tree, and graphs with many cycles."""
    rng = np.random.default_rng(N)
    column_of = rng.permutation(N).astype(np.int32)
    edges = np.zeros((N, N), np.int32)
    edges[np.arange(N), column_of] = 1
    if kind == "tree":
        for i in range(N // 2):
            edges[rng.integers(N), rng.integers(N)] = 1
    elif kind == "cycles":
        for _ in range(2 if N <= 64 else 1):
            edges[np.arange(N), rng.permutation(N)] = 1
    done = subprocess.run([program, "adopt"], input=np.array([N, 1], np.int32).tobytes() + edges.tobytes() + column_of.tobytes(),
                          capture_output=True, timeout=120, check=True)
    perm = np.frombuffer(done.stdout[8:], np.uint8)
    assert perm.tolist() == smallest_matching(edges, column_of.tolist())
