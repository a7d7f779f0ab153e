"""Sizes and values at which the kernels change their way of working, against the CPU oracle, bit for bit: whole warps and
slabs of rows, chunks and batches of matchings, 16-bit and 32-bit entries, one-word and two-step distances, the quick and
the ordinary division. (All results are whole numbers or defined operation by operation, so equality is the tolerance.)"""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_26845_b200 as ms
from paper_2605_26845_b200.workload import DEFAULT_MODEL, PROFILED_MODEL, bvn_capacity, random_matrices

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def random_schedule(B, K, N, seed, high):
    rng = np.random.default_rng(seed)
    perm = np.argsort(rng.random((B, K, N)), axis=2).astype(np.uint8)
    dur = rng.integers(0, high, size=(B, K)).astype(np.int32)
    return perm, dur


@pytest.mark.parametrize("K", [1, 31, 32, 33, 255, 256, 257, 520])
@pytest.mark.parametrize("N,B,high", [(1, 3, 50), (32, 3, 900), (33, 700, 900), (64, 3, 900), (64, 1600, 900), (65, 3, 90000),
                                      (128, 3, 900), (128, 320, 900), (192, 3, 90000), (193, 3, 900), (193, 3, 90000),
                                      (256, 3, 900), (256, 3, 90000)])
def test_scoring_at_the_edges_of_chunks_and_layouts(N, B, high, K):
    """Batches that are resident with 32-bit entries, that are not, and matrices that need them split over two CTAs."""
    few = 3
    D = random_matrices(few, N, seed=100 * N + K, high=high)
    perm, dur = random_schedule(few, K, N, N + K, 40)
    count = np.array([K, max(0, K - 1), K // 2], np.int32)
    which = np.arange(B) % few
    d, p, q, c = dev(D[which]), dev(perm[which]), dev(dur[which]), dev(count[which])
    for prefix in (False, True):
        s = ms.schedule_eval(d, p, q, c, PROFILED_MODEL, prefix=prefix)
        r = oracle.schedule_eval(D, perm, dur, count, PROFILED_MODEL, threads=8)
        for name in ms.SCORE_FIELDS + ("status",):
            assert (s[name].cpu().numpy() == r[name][which]).all(), name
        if prefix:
            rp = oracle.schedule_prefix_eval(D, perm, dur, count, PROFILED_MODEL, threads=8)
            for name in ("prefix_overlap_ns", "prefix_unserved_tokens"):
                assert (s[name].cpu().numpy() == rp[name][which]).all(), name


@pytest.mark.parametrize("N", [5, 33, 64, 100])
@pytest.mark.parametrize("offset", [1, 4, 15])
def test_scoring_of_a_schedule_at_any_address(N, offset):
    """The schedule is fetched in aligned groups of 16 bytes; its first byte may lie anywhere in one."""
    B, K = 4, 70
    D = random_matrices(B, N, seed=N, high=500)
    perm, dur = random_schedule(B, K, N, N, 30)
    count = np.array([70, 64, 33, 1], np.int32)
    room = torch.zeros(perm.size + offset, dtype=torch.uint8, device="cuda")
    p = room[offset:].view(B, K, N)
    p.copy_(dev(perm))
    perm[2, 5, 0] = perm[2, 5, 1] if N > 1 else 7            # one faulty schedule
    p[2, 5, 0] = p[2, 5, 1]
    s = ms.schedule_eval(dev(D), p, dev(dur), dev(count), DEFAULT_MODEL)
    r = oracle.schedule_eval(D, perm, dur, count, DEFAULT_MODEL, threads=4)
    assert list(r["status"]) == [0, 0, -1, 0]
    for name in ms.SCORE_FIELDS + ("status",):
        assert (s[name].cpu().numpy() == r[name]).all(), name


@pytest.mark.parametrize("N", [1, 2, 3, 4, 7])
@pytest.mark.parametrize("K", [1, 2, 3])
def test_scoring_of_schedules_shorter_than_a_group_of_bytes(N, K):
    """Several matrices lie in the first 16 bytes; the array may begin anywhere in them."""
    B = 9
    D = random_matrices(B, N, seed=N, high=500)
    perm, dur = random_schedule(B, K, N, 10 * N + K, 30)
    count = (np.arange(B) % (K + 1)).astype(np.int32)
    r = oracle.schedule_eval(D, perm, dur, count, DEFAULT_MODEL, threads=4)
    for offset in range(16):
        room = torch.full((perm.size + offset,), 255, dtype=torch.uint8, device="cuda")
        p = room[offset:].view(B, K, N)
        p.copy_(dev(perm))
        s = ms.schedule_eval(dev(D), p, dev(dur), dev(count), DEFAULT_MODEL)
        for name in ms.SCORE_FIELDS + ("status",):
            assert (s[name].cpu().numpy() == r[name]).all(), (name, offset)


@pytest.mark.parametrize("N", [4, 32, 33, 64, 72, 129, 200, 256])
@pytest.mark.parametrize("high", [65535, 65536, 1 << 20, (1 << 20) + 1, 1 << 28])
def test_greedy_at_the_edges_of_its_distances(N, high):
    """Largest entries on either side of 16 bits and of the one-word distances, and so large that a search leaves the
    range of a saturating one-word distance."""
    D = random_matrices(2, N, seed=N, high=high)
    D[0, 0, 0] = high
    D[1] = np.where(D[1] % 3 == 0, 0, D[1])
    K = 6 if N > 64 else 12
    g = ms.mw_decompose(dev(D), K, want_residual=True)
    r = oracle.mw_decompose(D, K, threads=8)
    assert (g.status.cpu().numpy() == r["status"]).all() and (g.count.cpu().numpy() == r["count"]).all()
    kk = np.arange(K)[None, :] < r["count"][:, None]
    assert (g.perm.cpu().numpy()[kk] == r["perm"][kk]).all() and (g.dur.cpu().numpy()[kk] == r["dur"][kk]).all()
    assert (g.extra.cpu().numpy() == r["residual"]).all()


@pytest.mark.parametrize("N,smooth,iters", [(3, 0.0, 1200), (8, 0.0, 400), (16, 1e300, 3), (64, 1e-300, 3), (7, 0.5, 40),
                                            (96, 0.5, 4), (97, 0.5, 4), (128, 0.5, 4), (160, 0.5, 3), (161, 0.5, 3)])
def test_scaling_at_the_ends_of_the_exponent_range_and_of_the_layouts(N, smooth, iters):
    """Without a perfect matching in the support some entries halve in every sweep, down to the subnormal numbers and zero."""
    D = random_matrices(3, N, seed=N, high=300, zero_frac=0.0 if smooth == 0.0 else 0.3)
    if smooth == 0.0:
        D[:] = D + 1
        D[:, :2, 1:] = 0                                     # two rows that reach the first column only
        D[2] = np.triu(D[2] + 1)
    g = ms.sinkhorn_scale(dev(D), iters, smooth, 20)
    r = oracle.sinkhorn_scale(D, iters, smooth, 20, threads=8)
    assert (g["status"].cpu().numpy() == r["status"]).all()
    for name in ("scaled", "fixed", "stretch", "row_err"):
        assert (g[name].cpu().numpy() == r[name]).all(), name


def test_path_takes_smaller_batches_and_refuses_larger_ones():
    path = ms.Path(40, 24, 10)
    for B, N in ((40, 24), (7, 24), (9, 11)):
        D = random_matrices(B, N, seed=B, high=400)
        d = dev(D)
        cap = path.k_bvn
        for overlap in (True, False):
            path.run(d, DEFAULT_MODEL, overlap=overlap)
            r = oracle.bvn_decompose(D, cap, threads=8)
            assert (path.bvn.count.cpu().numpy()[:B] == r["count"]).all()
            perm = path.bvn.perm.view(-1)[:B * cap * N].view(B, cap, N).cpu().numpy()
            kk = np.arange(cap)[None, :] < r["count"][:, None]
            assert (perm[kk] == r["perm"][kk]).all()
            rs = oracle.schedule_eval(D, r["perm"], r["coef"], r["count"], DEFAULT_MODEL, threads=8)
            for i, name in enumerate(ms.SCORE_FIELDS):
                assert (path.score_bvn[i, :B].cpu().numpy() == rs[name]).all(), name
    with pytest.raises(ms.MoeschedError):
        path.run(dev(random_matrices(41, 24, seed=1)))
    assert bvn_capacity(24) == path.k_bvn


@pytest.mark.parametrize("N", [65, 95, 96, 97, 128, 129, 159, 160, 161, 191, 192, 193, 223, 224, 225])
@pytest.mark.parametrize("high", [3, 2000, 90000])
def test_decomposers_at_the_edges_of_their_words(N, high):
    """One kernel per number of 32-column words a row set takes; tie-rich, 16-bit and 32-bit entries."""
    D = random_matrices(2, N, seed=N + high, high=high)
    for K, gpu, cpu, value in ((20, ms.mw_decompose, oracle.mw_decompose, "dur"), (60, ms.bvn_decompose, oracle.bvn_decompose, "coef")):
        g, r = gpu(dev(D), K), cpu(D, K, threads=2)
        assert (g.status.cpu().numpy() == r["status"]).all() and (g.count.cpu().numpy() == r["count"]).all()
        kk = np.arange(K)[None, :] < r["count"][:, None]
        assert (g.perm.cpu().numpy()[kk] == r["perm"][kk]).all() and (g.dur.cpu().numpy()[kk] == r[value][kk]).all()


@pytest.mark.parametrize("N", [229, 230, 231, 232, 233])
def test_where_one_cta_no_longer_holds_a_matrix(N):
    """Up to 232 ranks an int32 matrix and the state of its warp fit the shared memory of one CTA, above they take two: greedy
    with entries beyond 16 bits, Birkhoff without scratch."""
    D = random_matrices(3, N, seed=N, high=300000, zero_frac=0.4)
    for K, gpu, cpu, value in ((12, ms.mw_decompose, oracle.mw_decompose, "dur"),
                               (40, lambda d, k: ms.bvn_decompose(d, k, scratch=False), oracle.bvn_decompose, "coef")):
        g, r = gpu(dev(D), K), cpu(D, K, threads=3)
        assert (g.status.cpu().numpy() == r["status"]).all() and (g.count.cpu().numpy() == r["count"]).all()
        kk = np.arange(K)[None, :] < r["count"][:, None]
        assert (g.perm.cpu().numpy()[kk] == r["perm"][kk]).all() and (g.dur.cpu().numpy()[kk] == r[value][kk]).all()


@pytest.mark.parametrize("N", [33, 64, 65, 96, 97, 128, 129, 160, 161])
def test_decomposers_in_batches_that_are_not_resident(N):
    """A batch that does not fit half of the SMs' shared memory as int32 has its Birkhoff working copy in global memory and its
    greedy residual as 16-bit entries, here with some matrices that do not fit those."""
    D = random_matrices(5, N, seed=17 * N, high=3000)
    D[3] *= 50
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    which = np.arange(sms * (227 * 512 // (4 * N * N + 1024)) + 1) % 5
    for K, gpu, cpu, value in ((16, ms.mw_decompose, oracle.mw_decompose, "dur"), (70, ms.bvn_decompose, oracle.bvn_decompose, "coef")):
        g, r = gpu(dev(D[which]), K), cpu(D, K, threads=5)
        assert (g.status.cpu().numpy() == r["status"][which]).all() and (g.count.cpu().numpy() == r["count"][which]).all()
        kk = (np.arange(K)[None, :] < r["count"][:, None])[which]
        assert (g.perm.cpu().numpy()[kk] == r["perm"][which][kk]).all()
        assert (g.dur.cpu().numpy()[kk] == r[value][which][kk]).all()


@pytest.mark.parametrize("N", range(1, 13))
@pytest.mark.parametrize("kind", [dict(high=9000), dict(kind="ties"), dict(high=5, zero_frac=0.6)])
def test_birkhoff_decomposition_of_few_ranks(N, kind):
    """Up to eight ranks the matchings are read off bitmaps over all sets of columns, above they are searched for; one matrix per CTA
    and four, entries up to the largest sums, a matrix that is refused, and a budget that runs out."""
    few = 40
    D = random_matrices(few, N, seed=31 * N, **kind)
    D[0] = 0
    D[1] = 7
    D[2] *= (2**31 - 1) // max(1, int(max(D[2].sum(0).max(), D[2].sum(1).max())))
    D[3, N - 1, 0] = -1
    for B in (few, 16 * torch.cuda.get_device_properties(0).multi_processor_count + 3):
        which = np.arange(B) % few
        for K in (bvn_capacity(N), max(1, N // 2)):
            g, r = ms.bvn_decompose(dev(D[which]), K, want_aug=True), oracle.bvn_decompose(D, K, threads=8)
            assert (g.status.cpu().numpy() == r["status"][which]).all() and (g.count.cpu().numpy() == r["count"][which]).all()
            kk = (np.arange(K)[None, :] < r["count"][:, None])[which]
            assert (g.perm.cpu().numpy()[kk] == r["perm"][which][kk]).all()
            assert (g.dur.cpu().numpy()[kk] == r["coef"][which][kk]).all()
            assert (g.extra.cpu().numpy()[which != 3] == r["aug"][which][which != 3]).all()


def faulty_schedules(N, K, seed):
    """Schedules of K matchings, all but the first and the last with something wrong in them: destinations that do not exist at the
    edges of chunks of 32 and in a chunk that is not full, alone and in runs, and columns that only the matching before could mark."""
    perm, dur = random_schedule(1, K, N, seed, 40)
    none = [N] if N == 255 else [N, 255] if N < 255 else []

    def without_column(p, k, c):                       # row that had column c: the one of another row
        at = int(np.flatnonzero(p[k] == c)[0])
        p[k, at] = p[k, (at + 1) % N]

    out = [perm[0]]
    for k in (0, 15, 31, 32, 63, 64, K - 1):
        for bad in none:
            p = perm[0].copy()
            p[k, (7 * k) % N] = bad
            out.append(p)
        p = perm[0].copy()
        without_column(p, k, 0)
        out.append(p)
    for first, last in ((0, 31), (30, 33), (62, K - 1)):
        for bad in none:
            p = perm[0].copy()
            p[first:last + 1, N - 1] = bad             # every one spills into the next
            out.append(p)
            for k in range(first + 1, last + 1):       # ... whose only missing column is the first
                p[k] = perm[0, k]
                p[k, int(np.flatnonzero(p[k] == 0)[0])] = bad
            out.append(p.copy())
    for k in (10, 30, 31, 63):                         # one bad destination, then one column 0 missing
        for bad in none:
            p = perm[0].copy()
            p[k, 3 % N] = bad
            without_column(p, k + 1, 0)
            out.append(p)
    out.append(perm[0])
    return np.stack(out), np.repeat(dur, len(out), axis=0)


@pytest.mark.parametrize("N,B", [(33, 2100), (33, 2500), (62, 1500), (62, 1750), (64, 1500), (64, 1800), (65, 1100), (120, 600), (127, 500),
                                 (128, 500), (129, 400), (192, 200), (200, 200), (220, 90), (255, 90), (256, 90), (32, 90), (64, 90),
                                 (128, 90)])
def test_scoring_of_faulty_schedules(N, B):
    """Batches of 16-bit entries with one and two buffers for the marks, which may border on the next matching's, and a few of
    32-bit entries; sound schedules stand beside the faulty ones."""
    K = 70
    perm, dur = faulty_schedules(N, K, seed=N)
    F = len(perm)
    perm[F - 1, 60:] = 0                               # what lies beyond the count is not looked at
    count = np.full(F, K, np.int32)
    count[F - 1] = 60
    D = random_matrices(F, N, seed=3 * N, high=300)
    which = np.arange(B) % F
    which[:3] = 0, F - 1, 0
    d, p, q, c = dev(D[which]), dev(perm[which]), dev(dur[which]), dev(count[which])
    r = oracle.schedule_prefix_eval(D, perm, dur, count, PROFILED_MODEL, threads=8)
    rs = oracle.schedule_eval(D, perm, dur, count, PROFILED_MODEL, threads=8)
    assert (rs["status"] == np.r_[0, np.full(F - 2, ms.ST_BAD_INPUT), 0]).all()
    for prefix in (False, True):
        s = ms.schedule_eval(d, p, q, c, PROFILED_MODEL, prefix=prefix)
        for name in ms.SCORE_FIELDS + ("status",):
            assert (s[name].cpu().numpy() == rs[name][which]).all(), name
        if prefix:
            for name in ("prefix_overlap_ns", "prefix_unserved_tokens"):
                assert (s[name].cpu().numpy() == r[name][which]).all(), name
