"""What the Python binding hands to the library, seen from the host side (no GPU: the native call is recorded)."""
import contextlib

import numpy as np
import pytest
import torch

import paper_2605_26845_b200 as ms


@pytest.fixture
def calls(monkeypatch):
    """Native calls made by the binding, as (name, arguments without the stream); CPU tensors are let through."""
    made = []
    monkeypatch.setattr(ms, "_dev", lambda t, dtype, what: t)
    monkeypatch.setattr(ms, "_call", lambda name, device, *args: made.append((name, args)))
    return made


def schedule(B, N, K):
    return (torch.zeros((B, N, N), dtype=torch.int32), torch.zeros((B, K, N), dtype=torch.uint8),
            torch.zeros((B, K), dtype=torch.int32), torch.zeros(B, dtype=torch.int32))


@pytest.mark.parametrize("prefix", [False, True])
@pytest.mark.parametrize("form", ["five", "seven", "list", "slice"])
def test_scores_go_where_the_caller_wants_them(calls, form, prefix):
    """`out` may have rows to spare, be a sequence of tensors, or a part of a wider array."""
    B = 3
    out = {"five": torch.zeros((5, B), dtype=torch.int64), "seven": torch.zeros((7, B), dtype=torch.int64),
           "list": [torch.zeros(B, dtype=torch.int64) for _ in range(5)],
           "slice": torch.zeros((5, 2 * B), dtype=torch.int64)[:, B:]}[form]
    status = torch.zeros(B, dtype=torch.int32)
    res = ms.schedule_eval(*schedule(B, 4, 2), out=out, status=status, prefix=prefix)
    (name, args), = calls
    assert len(args) + 1 == len(ms._SIGNATURES[name])            # (the stream comes last)
    assert list(args[8:13]) == [out[i].data_ptr() for i in range(5)] and args[13] == status.data_ptr()
    for i, field in enumerate(ms.SCORE_FIELDS):
        assert res[field].data_ptr() == out[i].data_ptr() and res[field].shape == (B,)


def test_a_call_owns_its_model(calls):
    """The structure that the library reads belongs to the call that made it, whatever other models are used meanwhile, and
    holds the values that the dict has at the time of the call."""
    d, perm, dur, count = schedule(2, 4, 2)
    link = torch.tensor(400)
    model = dict(ms.DEFAULT_MODEL, link_gbps=link)
    made = {}
    for gbps in (400, 800):
        link.fill_(gbps)
        ms.schedule_eval(d, perm, dur, count, model)
        ms.schedule_order(d, perm, dur, count, model)
        ms.ideal_a2a(d, model)
        made[gbps] = [args[at] for (_, args), at in zip(calls[-3:], (7, 7, 3))]
    for other in range(300):
        ms.ideal_a2a(d, dict(ms.DEFAULT_MODEL, reconfig_ns=other))
    for gbps, structures in made.items():
        for m in structures:
            assert isinstance(m._obj, ms._Model) and m._obj.link_gbps == gbps
            assert m._obj.bytes_per_token == ms.DEFAULT_MODEL["bytes_per_token"]
    for value in (torch.tensor(500), np.array(500), np.int64(500), 500.0):     # with a hash or without
        ms.ideal_a2a(d, dict(ms.DEFAULT_MODEL, link_gbps=value))
        assert calls[-1][1][3]._obj.link_gbps == 500
    ms.ideal_a2a(d, dict(ms.DEFAULT_MODEL, link_gbps=400.9))
    ms.ideal_a2a(d, dict(ms.DEFAULT_MODEL, link_gbps=401))
    assert [args[3]._obj.link_gbps for _, args in calls[-2:]] == [400, 401]


class FakeStream:
    cuda_stream = 8


class FakeEvent:
    cuda_event = 16

    def record(self, stream=None):
        pass


@pytest.fixture
def path(calls, monkeypatch):
    monkeypatch.setattr(torch.cuda, "device", lambda dev: contextlib.nullcontext())
    monkeypatch.setattr(torch.cuda, "Stream", lambda *a, **k: FakeStream())
    monkeypatch.setattr(torch.cuda, "Event", lambda *a, **k: FakeEvent())
    return ms.Path(3, 4, 2, device="cpu", want_work=True)


def test_a_path_uses_the_buffers_that_it_has_at_the_time_of_the_call(calls, path):
    """Buffers are public: one that was replaced between two runs must neither be missed nor written to once it is gone."""
    demand = torch.zeros((3, 4, 4), dtype=torch.int32)

    def passed():
        path.run(demand)
        given = calls[-1][1][0]
        args = ms._PathArgs.from_address(given) if isinstance(given, int) else given._obj
        return {name: getattr(args, name) for name, _ in ms._PathArgs._fields_}

    def expected():
        return {"mw_perm": path.mw.perm, "bvn_perm": path.bvn.perm, "mw_dur": path.mw.dur, "mw_count": path.mw.count,
                "mw_status": path.mw.status, "mw_eval_status": path.eval_status_mw, "bvn_coef": path.bvn.dur,
                "bvn_count": path.bvn.count, "bvn_status": path.bvn.status, "bvn_eval_status": path.eval_status_bvn,
                "mw_work": path.mw.work, "bvn_work": path.bvn.work, "mw_scores": path.score_mw,
                "bvn_scores": path.score_bvn, "bvn_scratch": path.scratch}

    def check():
        got = passed()
        for name, tensor in expected().items():
            assert got[name] == (None if tensor is None else tensor.data_ptr()), name
        assert (got["k_mw"], got["k_bvn"], got["score_stride"]) == (path.k_mw, path.k_bvn, 3)

    check()
    old = []
    for holder, names in ((path.mw, ("perm", "dur", "count", "status", "work")), (path.bvn, ("perm", "dur", "count", "status", "work")),
                          (path, ("score_mw", "score_bvn", "eval_status_mw", "eval_status_bvn", "scratch"))):
        for name in names:
            old.append(getattr(holder, name))
            setattr(holder, name, torch.empty_like(old[-1]))
            check()
    path.mw.work = path.bvn.work = None
    check()
