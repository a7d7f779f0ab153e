"""Calls from several host threads at once: kernels that serve more than one size are launched with a different amount of shared
memory for each, and what a kernel may have is set for the whole process."""
import threading

import numpy as np
import pytest
import torch

import oracle
import paper_2605_26845_b200 as ms
from paper_2605_26845_b200.workload import random_matrices

pytestmark = pytest.mark.gpu


def greedy(N):
    d = torch.from_numpy(random_matrices(1, N, seed=N, high=900)).cuda()
    out = ms.mw_decompose(d, 1)
    ref = oracle.mw_decompose(d.cpu().numpy(), 1)
    return (lambda: ms.mw_decompose(d, 1, out=out)), (lambda: (out.perm.cpu().numpy() == ref["perm"]).all())


def scaling(N):
    d = torch.from_numpy(random_matrices(1, N, seed=N, high=900)).cuda()
    out = ms.sinkhorn_scale(d, 1)
    first = out["scaled"].clone()
    return (lambda: ms.sinkhorn_scale(d, 1, out=out)), (lambda: torch.equal(out["scaled"], first))


def ordering(K):
    d = torch.from_numpy(random_matrices(1, 4, seed=K, high=900)).cuda()
    perm = torch.arange(4, dtype=torch.uint8, device="cuda").expand(1, K, 4).contiguous()
    dur = torch.ones((1, K), dtype=torch.int32, device="cuda")
    count = torch.full((1,), K, dtype=torch.int32, device="cuda")
    got = {}

    def call():
        got.update(ms.schedule_order(d, perm, dur, count))
    return call, lambda: int(got["status"][0]) == 0 and got["order"][0].sort().values.tolist() == list(range(K))


@pytest.mark.parametrize("make,sizes", [(greedy, (112, 128)), (scaling, (130, 160)), (ordering, (40, 1024))])
def test_one_kernel_for_two_sizes_from_several_threads(make, sizes):
    pairs = [make(n) for n in sizes]
    torch.cuda.synchronize()
    errors, begin = [], threading.Barrier(2 * len(sizes))

    def work(call):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                begin.wait()
                for i in range(1500):
                    call()
                    if i % 100 == 99:
                        torch.cuda.current_stream().synchronize()
        except Exception as e:      # noqa: BLE001 (any error of a call counts)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(call,)) for call, _ in 2 * pairs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    assert all(ok() for _, ok in pairs)
