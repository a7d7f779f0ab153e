"""Timed workloads of the library: what its users have it do, through its public entry points.

listed() holds the named cases, draw() makes further ones of the same ranges. Demand matrices are token-routing
counts (see workload.py for the recipe; here it is drawn on the GPU): every rank routes `tokens` tokens to
top_k distinct experts each, the experts sit `per_rank` to a rank, so all row sums are equal, few pairs are heavy and
many are light or empty.

Kinds of work:
  path      both decompositions of a batch, each scored (Path.run, or its CUDA-graph form with graph=True)
  plan      choosing the circuits of the next all-to-alls: greedy matchings up to a budget, the score of every prefix,
            the best number of matchings, the order of the matchings and the reordered schedule
  sinkhorn  the paper's multiplicative route: Sinkhorn-Knopp scaling, then the Birkhoff decomposition of the scaled
            matrix, either real valued (real=True) or fixed point with durations in tokens and a score
  score     existing schedules under two compute models, next to the ideal all-to-all
  host      a stream of batches in pinned host memory through the double-buffered pipeline (two batches a pass)
"""
import math

import torch

import paper_2605_26845_b200 as ms
from paper_2605_26845_b200.workload import DEFAULT_MODEL, PROFILED_MODEL, bvn_capacity

UNSERVED_PRICE_NS = 100     # price of a token left unserved when a plan's budget is chosen
SCALE_BITS = 20             # fixed-point bits of the scaled matrices


def _case(kind, N, B, tokens, per_rank, top_k, traffic, budget=0, graph=False, real=False, schedule="", name=None):
    c = dict(kind=kind, N=N, B=B, tokens=tokens, per_rank=per_rank, top_k=top_k, traffic=traffic)
    if kind in ("path", "plan", "host") or schedule == "greedy":
        c["budget"] = budget or N
    if kind == "path":
        c["graph"] = graph
    if kind == "sinkhorn":
        c["real"] = real
    if kind == "score":
        c["schedule"] = schedule
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest batch: eight ranks, one expert each; a step is a few microsecond kernels and their launches
        _case("path", 8, 64, 4096, 1, 2, "zipf", name="path_n8_b64"),
        # a node pair with many layers and steps at once, replayed from a graph as a serving loop would
        _case("path", 16, 1024, 8192, 4, 6, "zipf", graph=True, name="path_n16_b1024_graph"),
        # the headline: thousands of 64-rank matrices
        _case("path", 64, 4096, 16384, 4, 8, "zipf", name="path_n64_b4096"),
        # 128 ranks, every source rank with preferences of its own
        _case("path", 128, 1024, 8192, 4, 8, "dirichlet", name="path_n128_b1024"),
        # the largest domain the library takes; most pairs exchange nothing
        _case("path", 256, 256, 4096, 4, 8, "sparse", name="path_n256_b256"),
        # a handful of layers on an odd number of ranks: too few matrices to fill the GPU
        _case("path", 100, 3, 8192, 4, 8, "dirichlet", name="path_n100_b3"),
        # one all-to-all planned on line, between two layers: nothing but latency
        _case("plan", 64, 1, 16384, 4, 8, "zipf", budget=16, name="plan_n64_b1"),
        # plans for all layers of a step with very large token counts (entries beyond 16 bits)
        _case("plan", 72, 60, 1 << 22, 4, 8, "zipf", name="plan_n72_b60_wide"),
        # the paper's preprocessing, schedule in tokens
        _case("sinkhorn", 64, 1024, 16384, 4, 8, "zipf", name="sinkhorn_fixed_n64_b1024"),
        # the same with real coefficients, one rank more than a warp has lanes
        _case("sinkhorn", 33, 512, 8192, 4, 6, "zipf", real=True, name="sinkhorn_real_n33_b512"),
        # what-if scoring of complete Birkhoff schedules: the schedule is read from memory, a gigabyte of it
        _case("score", 64, 4096, 16384, 4, 8, "zipf", schedule="bvn", name="score_n64_b4096"),
        # batches that arrive in and return to host memory
        _case("host", 64, 512, 16384, 4, 8, "zipf", name="host_n64_b512"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choices(("path", "plan", "sinkhorn", "score", "host"), (9, 4, 3, 2, 2))[0]
    schedule = rng.choice(("bvn", "greedy")) if kind == "score" else ""
    top_n = 256 if kind in ("path", "plan") or schedule == "greedy" else 96
    N = _log_int(rng, 4, top_n)
    # entries of a batch; bounded more tightly where a matrix is costlier, so that no draw passes the largest listed case
    entries = 1 << 21 if kind == "host" or N > 128 else 1 << 23
    B = _log_int(rng, 1, max(1, min(4096, entries // (N * N))))
    tokens = _log_int(rng, 1024, 32768)
    per_rank = rng.choice((1, 2, 4))
    if kind != "sinkhorn" and rng.random() < 0.15:   # entries beyond 16 bits, column sums still within 31
        tokens = min(tokens << 8, (1 << 31) // (N * per_rank) - 1)
    top_k = rng.randint(1, min(8, max(1, N * per_rank // 4)))
    traffic = rng.choice(("zipf", "zipf", "dirichlet", "sparse"))
    budget = rng.choice((max(1, N // 8), max(1, N // 4), N))
    return _case(kind, N, B, tokens, per_rank, top_k, traffic, budget=budget, graph=kind == "path" and rng.random() < 0.3,
                 real=rng.random() < 0.5, schedule=schedule)


# ---- demand matrices -----------------------------------------------------------------------------------------

def _popularity(case, nb, gen):
    """Expert probabilities per matrix and source rank, [nb, N, E] float64."""
    N, E = case["N"], case["N"] * case["per_rank"]
    dev = gen.device

    def uniform(*shape):
        return torch.rand(shape, generator=gen, device=dev, dtype=torch.float64).clamp_(min=1e-12)

    if case["traffic"] == "dirichlet":     # every source rank has its own favourites, some experts are hot for all
        p = -torch.log(uniform(nb, N, E)) * uniform(nb, N, E) ** (1 / 0.3)
        p = p / p.sum(-1, keepdim=True) + 1e-9
        p = torch.where(uniform(nb, 1, E) < 0.05, 10 * p, p)
    else:                                  # Zipf popularity in an order of its own for every matrix
        skew = 1.4 if case["traffic"] == "sparse" else 1.2
        base = torch.arange(1, E + 1, device=dev, dtype=torch.float64) ** -skew
        p = base[torch.argsort(uniform(nb, E), dim=-1)][:, None, :].expand(nb, N, E)
        if case["traffic"] == "sparse":    # a source rank reaches about four destinations in ten
            allow = uniform(nb, N, N) < 0.4
            idx = torch.arange(N, device=dev)
            for extra in range(-(-case["top_k"] // case["per_rank"])):   # enough ranks to host top_k experts
                allow[:, idx, (idx + extra) % N] = True
            p = torch.where(allow.repeat_interleave(case["per_rank"], dim=-1), p, torch.zeros_like(p))
    return p / p.sum(-1, keepdim=True)


def _selections(p, tokens, top_k, gen):
    """Tokens per expert, [R, E]: every token takes top_k distinct experts by systematic sampling from the inclusion
    probabilities min(1, c p); the counts follow from how many of the tokens' offsets fall into each arc between the
    fractional parts of the cumulative probabilities (a chain of binomials)."""
    R, E = p.shape
    capped = torch.zeros_like(p, dtype=torch.bool)
    for _ in range(top_k + 1):
        c = (top_k - capped.sum(-1, keepdim=True)) / p.masked_fill(capped, 0).sum(-1, keepdim=True).clamp(min=1e-300)
        capped |= c * p >= 1
    q = torch.where(capped, torch.ones_like(p), (c * p).clamp(max=1))
    cum = torch.cumsum(q, -1)
    cum[:, -1] = top_k
    whole = torch.floor(cum)
    at, order = torch.sort(cum - whole, dim=-1)
    mass = torch.ones(R, device=p.device, dtype=p.dtype)
    left = torch.full_like(mass, tokens)
    below = torch.zeros_like(p)
    edge = torch.zeros_like(mass)
    for a in range(E):
        share = ((at[:, a] - edge) / mass.clamp(min=1e-300)).clamp(0, 1)
        n = torch.binomial(left, share, generator=gen)
        left = left - n
        mass = mass - (at[:, a] - edge)
        edge = at[:, a]
        below[:, a] = tokens - left
    upto = tokens * whole + torch.zeros_like(p).scatter_(-1, order, below)
    upto[:, -1] = tokens * top_k
    return torch.diff(upto, dim=-1, prepend=torch.zeros(R, 1, device=p.device, dtype=p.dtype))


def _demand(case, seed):
    B, N = case["B"], case["N"]
    E = N * case["per_rank"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty((B, N, N), dtype=torch.int32, device="cuda")
    chunk = max(1, (1 << 25) // (N * E))
    for b in range(0, B, chunk):
        nb = min(chunk, B - b)
        p = _popularity(case, nb, gen)
        counts = _selections(p.reshape(nb * N, E), case["tokens"], case["top_k"], gen)
        out[b:b + nb] = counts.clamp_(min=0).reshape(nb, N, N, case["per_rank"]).sum(-1).to(torch.int32)
    return out


def _schedule(B, N, k):
    """A caller-made schedule; zeroed, since the library writes the first count[b] matchings only."""
    return ms.Schedule(perm=torch.zeros((B, k, N), dtype=torch.uint8, device="cuda"),
                       dur=torch.zeros((B, k), dtype=torch.int32, device="cuda"),
                       count=torch.zeros(B, dtype=torch.int32, device="cuda"),
                       status=torch.zeros(B, dtype=torch.int32, device="cuda"))


def _zero(path):
    for t in path.outputs():
        t.zero_()
    return path


# ---- one case ------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind, B, N = case["kind"], case["B"], case["N"]
    state = dict(case=case, demand=_demand(case, seed))
    if kind == "path":
        state["path"] = _zero(ms.Path(B, N, case["budget"]))
    elif kind == "plan":
        state["out"] = _schedule(B, N, case["budget"])
    elif kind == "sinkhorn" and not case["real"]:
        state["out"] = _schedule(B, N, bvn_capacity(N))
        state["scratch"] = torch.empty(ms.bvn_scratch_bytes(B, N), dtype=torch.uint8, device="cuda")
    elif kind == "score":
        k = case["budget"] if case["schedule"] == "greedy" else bvn_capacity(N)
        decompose = ms.mw_decompose if case["schedule"] == "greedy" else ms.bvn_decompose
        state["schedule"] = decompose(state["demand"], k, out=_schedule(B, N, k))
    elif kind == "host":
        state["pipe"] = ms.HostPipeline(B, N, case["budget"])
        for path in state["pipe"].paths:
            _zero(path)
        first, second = state.pop("demand"), _demand(case, seed + (1 << 32))
        state["batches"] = [first.cpu().pin_memory(), second.cpu().pin_memory()]
    return state


def run(state):
    case = state["case"]
    kind, N = case["kind"], case["N"]
    if kind == "path":
        path = state["path"]
        (path.run_graph if case["graph"] else path.run)(state["demand"])
        return path.outputs()
    if kind == "plan":
        d = state["demand"]
        s = ms.mw_decompose(d, case["budget"], out=state["out"])
        score = ms.schedule_eval(d, s.perm, s.dur, s.count, prefix=True)
        best = ms.best_budget(s.count, score["prefix_overlap_ns"], score["prefix_unserved_tokens"], UNSERVED_PRICE_NS)
        order = ms.schedule_order(d, s.perm, s.dur, s.count, PROFILED_MODEL)
        perm, dur = ms.schedule_permute(s.perm, s.dur, order["order"])
        return [s.perm, s.dur, s.count, s.status, score, best, order, perm, dur]
    if kind == "sinkhorn":
        scaled = ms.sinkhorn_scale(state["demand"], scale_bits=SCALE_BITS)
        if case["real"]:
            s = ms.bvn_real_decompose(scaled["scaled"])
            # entries beyond a matrix's count are not written: a reader of the schedule masks them
            used = torch.arange(s["lam"].shape[1], device="cuda") < s["count"][:, None]
            s["lam"] = torch.where(used, s["lam"], 0.0)
            s["perm"] = torch.where(used[:, :, None], s["perm"], 0)
            return [scaled, s]
        s = ms.bvn_decompose(scaled["fixed"], out=state["out"], scratch=state["scratch"])
        dur = ms.sinkhorn_durations(s.dur, s.count, scaled["stretch"], SCALE_BITS)
        score = ms.schedule_eval(state["demand"], s.perm, dur, s.count)
        return [scaled, s.perm, s.dur, s.count, s.status, dur, score]
    if kind == "score":
        s = state["schedule"]
        return [ms.schedule_eval(state["demand"], s.perm, s.dur, s.count, model) for model in (DEFAULT_MODEL, PROFILED_MODEL)] \
            + [ms.ideal_a2a(state["demand"])]
    pipe = state["pipe"]
    slots = [pipe.submit(batch) for batch in state["batches"]]
    return [pipe.result(slot) for slot in slots]


def work(case):
    """Inputs read once and outputs written once. The number of matchings depends on the data: a greedy schedule has
    about N of them, a complete Birkhoff schedule about as many as the matrix has entries. Operations: a greedy
    matching looks at every entry of the residual, a Birkhoff matching touches each row a few times."""
    kind, B, N = case["kind"], case["B"], case["N"]
    matrix = 4 * N * N
    kg = min(case.get("budget", N), N)
    kb = int((0.4 if case["traffic"] == "sparse" else 0.95) * bvn_capacity(N))
    greedy, bvn = kg * (N + 4), kb * (N + 4)
    if kind in ("path", "host"):
        return {"bytes": B * (matrix + greedy + bvn) * (2 if kind == "host" else 1),
                "flops": B * (kg * 2 * N * N + kb * 8 * N) * (2 if kind == "host" else 1)}
    if kind == "plan":
        return {"bytes": B * (matrix + 2 * greedy + 20 * kg), "flops": B * kg * 2 * N * N}
    if kind == "sinkhorn":
        return {"bytes": B * (matrix + 3 * matrix + bvn + 4 * kb), "flops": B * (20 * 4 * N * N + kb * 8 * N)}
    return {"bytes": B * (matrix + (greedy if case["schedule"] == "greedy" else bvn)), "flops": 0}


def tolerance(case):
    """Schedules and scores are whole numbers; the doubles are defined operation by operation, in a fixed order."""
    return "exact"
