"""What a user of the library has it do, as cases that can be timed.

A case is a dict of plain values.  `do` names the kind of work:

  sweep    a batch of placements scored against one trace, or several in one pass, and the best k of them
           (Context.eval_placements / eval_placements_multi, Context.topk)
  host     the same batch with host arrays in and out (Context.eval_placements_host)
  inspect  a few placements looked at closely: per-request times, unserved requests by model, latency
           histogram and percentiles, score
  rank     records of a finished sweep ranked again: by hits, by composite score, tail percentiles
  replan   the whole placer on a new request window: load the trace, prune the configurations, partition

and `space` the placements and the workload they are scored on:

  tiny     one model, tensor parallelism 1, 2, 4 on 4 devices
  node     one model, the ten (tp, pp) strategies on one node of 8 devices, every multiset in which the
           instances of a strategy share a batch cap
  multi    three models (1x, 1.9x, 9x), sampled placements of a cluster of 16 to 128 devices
  paper    the paper's own shape: three models, 24 devices, tables from its throughput decay function,
           gamma arrivals, decode lengths and SLO factors of its Table I (71 classes)
  large    placements of 33 to 128 instances on a modelled cluster of 1,024 devices
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_2509_06362_b200 as maaso

WMAX = 64
BATCHES = (1, 2, 4, 8, 16, 32, 64)
STRATEGIES = ((1, 1), (2, 1), (1, 2), (4, 1), (2, 2), (1, 4), (8, 1), (4, 2), (2, 4), (1, 8))
OPTIMISTIC, FROZEN, MAXGAP, QUEUES = 1, 2, 4, 8  # maaso_eval_opts.flags

INTERACTIVE, CHAT = (500_000, 50_000, None), (2_000_000, 150_000, None)
DOCUMENT, BATCH = (None, None, 180_000_000), (30_000_000, None, 600_000_000)


def listed():
    return [
        # The smallest call: every placement on four devices against a short trace.  Latency and launches.
        dict(name="tiny sweep", do="sweep", space="tiny", n_cand=143, budget=4, n_req=500, rate=8.0, traces=1,
             flags=0, masked=False, k=64),
        # One node searched exhaustively, the ordinary planning call.
        dict(name="node sweep", do="sweep", space="node", n_cand=10_864, budget=8, n_req=10_000, rate=16.0, traces=1,
             flags=0, masked=False, k=64),
        # The largest: a sampled cluster of 32 devices under a load that most placements cannot carry.
        dict(name="multi-model sweep", do="sweep", space="multi", n_cand=100_000, budget=32, n_req=100_000, rate=64.0,
             traces=1, flags=0, masked=False, k=64),
        # A big cluster split in two: each placement is scored on the requests of its own sub-cluster.
        dict(name="sub-cluster sweep", do="sweep", space="multi", n_cand=30_011, budget=128, n_req=40_007, rate=256.0,
             traces=1, flags=0, masked=True, k=256),
        # The load sweep: the same placements under sixteen arrival rates at once, bursty arrivals, the
        # distributor with its optimistic estimate.
        dict(name="load sweep, optimistic", do="sweep", space="node", n_cand=10_864, budget=8, n_req=10_000, rate=1.0,
             traces=16, flags=OPTIMISTIC, masked=False, k=64),
        # The paper's own workload.
        dict(name="paper sweep", do="sweep", space="paper", n_cand=2_000, budget=24, n_req=17_000, rate=17_000 / 3600,
             traces=1, flags=0, masked=False, k=64),
        # The same under the engine with a queue in front of every instance.
        dict(name="paper sweep, queues", do="sweep", space="paper", n_cand=1_999, budget=24, n_req=17_000,
             rate=17_000 / 3600, traces=1, flags=QUEUES, masked=False, k=64),
        # Placements of 33 to 128 instances.
        dict(name="large placements", do="sweep", space="large", n_cand=2_000, budget=1024, n_req=10_000, rate=400.0,
             traces=1, flags=0, masked=False, k=64),
        # A batch that a host program holds in its own arrays.
        dict(name="host arrays", do="host", space="multi", n_cand=3_001, budget=32, n_req=5_003, rate=64.0, flags=0),
        # The best placements of a sweep looked at closely.
        dict(name="inspection", do="inspect", space="multi", n_cand=64, budget=32, n_req=20_000, rate=24.0, flags=0),
        # The records of a million placements ranked.
        dict(name="ranking", do="rank", n_cand=1_000_000, k=64),
        # The placer itself: what runs whenever a new request window has been collected.
        dict(name="replan", do="replan", space="paper", gpus=24, n_req=17_000, rate=17_000 / 3600),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(("sweep",) * 7 + ("host", "inspect", "rank", "replan"))
    if do == "rank":
        return dict(do=do, n_cand=_log_int(rng, 300, 1_000_000), k=_log_int(rng, 1, 1024))
    if do == "replan":
        gpus = rng.randint(6, 32)
        return dict(do=do, space="paper", gpus=gpus, n_req=_log_int(rng, 1_000, 17_000),
                    rate=gpus * rng.uniform(0.1, 0.4))
    if do == "inspect":
        return dict(do=do, space="multi", n_cand=_log_int(rng, 8, 256), budget=rng.choice((16, 32, 64)),
                    n_req=_log_int(rng, 1_000, 30_000), rate=rng.uniform(10.0, 80.0), flags=rng.choice((0, 0, OPTIMISTIC)))
    if do == "host":
        return dict(do=do, space="multi", n_cand=_log_int(rng, 100, 10_000), budget=rng.choice((16, 32, 64)),
                    n_req=_log_int(rng, 500, 10_000), rate=rng.uniform(20.0, 100.0), flags=rng.choice((0, 0, OPTIMISTIC)))
    space = rng.choice(("tiny", "node", "node", "multi", "multi", "multi", "paper", "paper", "large"))
    # mostly the default engine and the two estimates; now and then one of the other readings
    flags = rng.choice((0,) * 6 + (OPTIMISTIC,) * 2 + (FROZEN, MAXGAP, QUEUES))
    c = dict(do=do, space=space, budget=8, traces=1, flags=flags, masked=False, k=rng.choice((1, 10, 64, 64, 500)))
    if space == "tiny":
        c.update(n_cand=rng.randint(20, 143), budget=4, n_req=_log_int(rng, 200, 5_000), rate=rng.uniform(2.0, 30.0))
    elif space == "node":
        c.update(n_cand=_log_int(rng, 200, 10_864), n_req=_log_int(rng, 500, 20_000), rate=_log_int(rng, 2, 64) * 1.0)
        if rng.random() < 0.3:
            c.update(traces=rng.randint(2, 16), rate=1.0)
    elif space == "multi":
        budget = rng.choice((16, 32, 48, 64, 128))
        c.update(n_cand=_log_int(rng, 200, 60_000), budget=budget, n_req=_log_int(rng, 1_000, 60_000),
                 rate=budget * rng.uniform(0.5, 2.5), masked=rng.random() < 0.3)
    elif space == "paper":
        c.update(n_cand=_log_int(rng, 200, 6_000), budget=24, n_req=_log_int(rng, 2_000, 17_000),
                 rate=rng.uniform(2.0, 8.0))
    else:
        c.update(n_cand=_log_int(rng, 100, 2_000), budget=1024, n_req=_log_int(rng, 1_000, 10_000),
                 rate=rng.uniform(200.0, 600.0))
    # no drawn case costs more than the largest listed one
    most = 1_000_000_000 if flags in (0, OPTIMISTIC) else 250_000_000
    c["n_req"] = max(200, min(c["n_req"], most // (c["n_cand"] * c["traces"])))
    return c


# ---- inputs ---------------------------------------------------------------------------------------------
def _half_up(x):
    return np.floor(x + 0.5).astype(np.int32)


def _profile(space, rng):
    """Latency tables: prefill and decode-step times by model, strategy and running count."""
    strategies = ((1, 1), (2, 1), (4, 1)) if space == "tiny" else STRATEGIES
    scale = np.array((1.0,) if space in ("tiny", "node") else (1.0, 1.9, 9.0))[:, None, None]
    tp = np.array([s[0] for s in strategies], dtype=np.float64)[None, :, None]
    pp = np.array([s[1] for s in strategies], dtype=np.float64)[None, :, None]
    w = np.arange(1, WMAX + 1, dtype=np.float64)[None, None, :]
    bubble = 1.0 + 0.15 * (pp - 1)
    jitter = 0.05 if space in ("node", "multi", "large") else 0.0
    shape = (scale.shape[0], len(strategies))
    u = rng.uniform(1 - jitter, 1 + jitter, size=shape + (WMAX + 2,))
    if space == "paper":  # the throughput decay function of the paper's profiler
        t0 = tp / (0.009 * scale) / bubble
        step = 1e6 / (t0 * (1.0 - (0.08 + 0.02 * np.log2(tp * pp)) * np.log(1.0 + w)))
    else:
        step = scale * (9000.0 / tp + 150.0 * w) * bubble * u[:, :, :WMAX]
    return {
        "n_models": shape[0], "n_strategies": shape[1], "wmax": WMAX,
        "devices": np.array([a * b for a, b in strategies], dtype=np.int32),
        "min_devices": np.array((1, 1, 4)[:shape[0]], dtype=np.int32),
        "prefill_base_us": _half_up((scale * (2000.0 / tp) * bubble)[:, :, 0] * u[:, :, WMAX]),
        "prefill_q16": _half_up((scale * (0.12 / tp) * bubble)[:, :, 0] * u[:, :, WMAX + 1] * 65536.0),
        "step_us": np.maximum(1, _half_up(step)),
    }


def _classes(space, profile):
    if space == "paper":  # per-token budgets: SLO factors 0.80 to 1.50 of the level-1 step of model 0
        rows = [(None, int(f * profile["step_us"][0, 0, 0] + 0.5), None) for f in np.arange(0.80, 1.505, 0.01)]
    else:
        rows = [INTERACTIVE, CHAT, DOCUMENT] + ([BATCH] if space == "large" else [])
    out = np.zeros(len(rows), dtype=maaso.SLO_DTYPE)
    for k, row in enumerate(rows):
        out[k] = tuple(-1 if x is None else x for x in row)
    return out


def _trace(space, n, rate, rng, cv=1.0):
    """n requests, gamma inter-arrival gaps with mean 1/rate s and coefficient of variation cv."""
    t = np.zeros(n, dtype=maaso.REQUEST_DTYPE)
    shape = 1.0 / (cv * cv)
    t["arrival_us"] = np.floor(np.cumsum(rng.gamma(shape, 1.0 / (rate * shape), size=n)) * 1e6)
    t["in_tokens"] = np.clip(rng.lognormal(6.0, 0.8, size=n) + 0.5, 16, 4096)
    if space == "paper":  # half short decodes with tight factors, half long ones with loose factors
        loose = rng.random(n) < 0.5
        t["out_tokens"] = np.where(loose, rng.integers(600, 1001, size=n), rng.integers(300, 501, size=n))
        t["cls"] = np.where(loose, rng.integers(40, 71, size=n), rng.integers(0, 21, size=n))
        t["model"] = rng.integers(0, 3, size=n)
        return t
    mix = np.cumsum({"large": (0.45, 0.27, 0.18, 0.10)}.get(space, (0.7, 0.2, 0.1) if cv > 1 else (0.5, 0.3, 0.2)))
    t["cls"] = np.minimum(np.searchsorted(mix, rng.random(n), side="right"), len(mix) - 1)
    if space in ("multi", "large"):
        t["model"] = np.minimum(np.searchsorted((0.6, 0.9, 1.0), rng.random(n), side="right"), 2)
    out = np.clip(rng.lognormal(4.5, 1.0, size=n) + 0.5, 1, 2048).astype(np.int64)
    t["out_tokens"] = np.where(t["cls"] == 2, rng.integers(2048, 8193, size=n), out)
    return t


def _words(model, strategy, batch):
    return model | (strategy << 4) | (batch << 12)


@functools.lru_cache(maxsize=None)
def _enumerated(space):
    """All placements of the one-model spaces, as lists of instance words."""
    out = []
    if space == "tiny":
        types = [(s, b) for s in range(3) for b in (1, 4, 8, 16)]
        for size in range(1, 5):
            for combo in itertools.combinations_with_replacement(types, size):
                if sum(1 << s for s, _ in combo) <= 4:
                    out.append([_words(0, s, b) for s, b in combo])
        return out
    cost = [a * b for a, b in STRATEGIES]

    def rec(s, left, used):
        if s == len(cost):
            for caps in itertools.product(BATCHES, repeat=len(used)):
                if used:
                    out.append([_words(0, k, b) for (k, n), b in zip(used, caps) for _ in range(n)])
            return
        for n in range(left // cost[s] + 1):
            rec(s + 1, left - n * cost[s], used + ([(s, n)] if n else []))

    rec(0, 8, [])
    return out


def _sampled(n, budget, profile, seed, at_least, stop_p):
    """Placements drawn instance by instance, uniformly among the types that still fit, until a coin or the
    budget ends it; instances sorted by (model, strategy, batch cap).  Returns offsets and words (CUDA)."""
    dev = profile["devices"]
    types = [(int(dev[s]), m, s, b) for m in range(profile["n_models"]) for s in range(len(dev))
             if dev[s] >= profile["min_devices"][m] for b in BATCHES]
    types.sort()
    cost = torch.tensor([t[0] for t in types], device="cuda")
    word = torch.tensor([_words(*t[1:]) for t in types], device="cuda")
    key = torch.tensor([(t[1] << 16) | (t[2] << 8) | t[3] for t in types], device="cuda")
    fits = torch.searchsorted(cost, torch.arange(budget + 1, device="cuda"), right=True)
    g = torch.Generator(device="cuda").manual_seed(seed)
    pool = n if at_least <= 1 else 3 * n + 64
    left = torch.full((pool,), budget, device="cuda")
    ids, picks = torch.arange(pool, device="cuda"), []
    for _ in range(128):
        ids = ids[fits[left[ids]] > 0]
        if not len(ids):
            break
        t = (torch.rand(len(ids), generator=g, device="cuda", dtype=torch.float64) * fits[left[ids]]).long()
        picks.append((ids, t))
        left[ids] -= cost[t]
        ids = ids[torch.rand(len(ids), generator=g, device="cuda") >= stop_p]
    cand, typ = torch.cat([p[0] for p in picks]), torch.cat([p[1] for p in picks])
    count = torch.bincount(cand, minlength=pool)
    keep = torch.nonzero(count >= at_least).flatten()[:n]
    rank = torch.full((pool,), -1, device="cuda")
    rank[keep] = torch.arange(len(keep), device="cuda")
    cand, typ = rank[cand], typ[rank[cand] >= 0]
    cand = cand[cand >= 0]
    order = torch.argsort((cand << 24) | key[typ], stable=True)
    offsets = torch.cat([torch.zeros(1, dtype=torch.long, device="cuda"), torch.cumsum(count[keep], 0)])
    return offsets.int(), word[typ[order]].int()


def _placements(case, profile, seed):
    space = case["space"]
    if space in ("tiny", "node"):
        every = _enumerated(space)
        n = min(case["n_cand"], len(every))
        rows = [every[i * len(every) // n] for i in range(n)]
        offsets = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
        words = np.fromiter(itertools.chain.from_iterable(rows), dtype=np.int32)
        return torch.from_numpy(offsets).cuda(), torch.from_numpy(words).cuda()
    large = space == "large"
    return _sampled(case["n_cand"], case["budget"], profile, seed, 33 if large else 1, 0.015 if large else 0.125)


def _records(n, seed):
    """Records of a finished sweep: a few invalid placements, hit counts that pile up where the good ones are."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def u():
        return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)

    counted = 100_000
    served = (counted * u() ** 2).long()
    hit = (served * (0.3 + 0.7 * u())).long()
    ttft = (served * (50_000 + 2_000_000 * u() ** 3)).long()
    r = torch.zeros((n, 16), dtype=torch.long, device="cuda")
    r[:, 0] = counted << 32
    r[:, 1] = served | (hit << 32)
    r[:, 2] = (counted - served) | ((served - hit) << 32)
    r[:, 7] = ttft
    r[:, 8] = (5_000_000 * u()).long()
    r[:, 9] = ttft + served * 9_000_000
    r[:, 10] = (90_000_000 * u()).long()
    r[:, 11] = 1_560_000_000 + (90_000_000 * u()).long()
    r[:, 12] = served * 150
    r[:, 13] = (u() * 2**62).long()
    r[:, 14] = counted + hit
    bad = u() < 0.01
    r[bad] = 0
    r[bad, 0] = 1
    # histograms of the time to first token: counts around a mean bin
    mean = 8 + 24 * u()[:, None]
    bins = torch.arange(64, device="cuda", dtype=torch.float64)[None, :]
    hist = (served[:, None] * torch.exp(-((bins - mean) / 4.0) ** 2) / 7.0).int()
    hist[bad] = 0
    return r.view(torch.uint8), hist


def _inputs(case, seed):
    space, rng = case["space"], np.random.default_rng(seed)
    profile = _profile(space, rng)
    n_traces = case.get("traces", 1)
    rates = [case["rate"]] if n_traces == 1 else [case["rate"] * 64.0 ** (j / (n_traces - 1)) for j in range(n_traces)]
    cv = 2.0 if space == "paper" else (4.0 if n_traces > 1 else 1.0)
    return profile, _classes(space, profile), [_trace(space, case["n_req"], r, rng, cv) for r in rates]


def prepare(case, seed):
    do = case["do"]
    s = {"do": do, "case": case, "ctx": maaso.Context(torch.cuda.current_device())}
    if do == "rank":
        s["records"], s["hist"] = _records(case["n_cand"], seed)
        return s
    profile, classes, traces = _inputs(case, seed)
    s["ctx"].load_profile(profile)
    if do == "replan":
        s["requests"], s["classes"], s["n_strategies"] = traces[0], classes, profile["n_strategies"]
        if case["space"] == "paper":  # two kinds of users, tight and loose, as masks need at most 32 classes
            loose = traces[0]["cls"] >= 40
            traces[0]["cls"] = np.where(loose, 2 + (traces[0]["cls"] - 40) // 16, traces[0]["cls"] // 11)
            s["classes"] = classes[[5, 15, 48, 64]]
        return s
    s["traces"] = [s["ctx"].load_trace(t, classes) for t in traces]
    s["offsets"], s["inst"] = _placements(case, profile, seed)
    if do == "host":
        s["offsets"], s["inst"] = (x.cpu().numpy().view(np.uint32) for x in (s["offsets"], s["inst"]))
    if case.get("masked"):  # placements of the interactive and chat sub-cluster, and of the document one
        s["mask"] = torch.where(torch.arange(case["n_cand"], device="cuda") % 3 < 2, 3, 4).int()
    if do == "inspect":
        s["look"] = np.arange(0, case["n_cand"], 2, dtype=np.uint32)
    return s


# ---- one pass -------------------------------------------------------------------------------------------
SCORE = dict(alpha=4.0, beta=0.3, gamma_t=20_000.0, gamma_l=10.0)


def run(s):
    case, ctx = s["case"], s["ctx"]
    if s["do"] == "rank":
        scores = ctx.score(s["records"], **SCORE)
        idx, rec = ctx.topk(s["records"], case["k"])
        idx_s, rec_s = ctx.topk_scores(s["records"], scores, case["k"])
        tails = ctx.ttft_percentiles(s["hist"], (500, 900, 990))
        return {"scores": scores, "idx": idx, "rec": rec.view(torch.int64), "idx_s": idx_s,
                "rec_s": rec_s.view(torch.int64), "tails": tails}
    if s["do"] == "replan":
        trace = ctx.load_trace(s["requests"], s["classes"])
        configs = ctx.prune_configs(trace, s["n_strategies"], BATCHES)
        plan = ctx.partition(trace, 0b0011, 0b1100, case["gpus"], configs, **SCORE, baseline=True)
        ctx.free_trace(trace)
        return {"configs": np.array(configs, dtype=np.int64), "g_t": plan["g_t"], "g_l": plan["g_l"],
                "phi": plan["phi"], "inst_t": plan["inst_t"], "inst_l": plan["inst_l"]}
    if s["do"] == "host":
        out = ctx.eval_placements_host(s["traces"][0], s["offsets"], s["inst"], case["budget"], flags=case["flags"])
        return {"records": out.view(np.int64).reshape(-1, 16)}
    if s["do"] == "inspect":
        n = case["n_cand"]
        rejected = torch.empty((n, 16), dtype=torch.int32, device="cuda")
        hist = torch.empty((n, 64), dtype=torch.int32, device="cuda")
        out, dumps = ctx.eval_placements(s["traces"][0], s["offsets"], s["inst"], case["budget"], flags=case["flags"],
                                         dump_idx=s["look"], rejected_by_model=rejected, ttft_hist=hist)
        return {"records": out.view(torch.int64), "rejected": rejected, "hist": hist, "dumps": dumps,
                "tails": ctx.ttft_percentiles(hist, (500, 900, 950, 990)), "scores": ctx.score(out, **SCORE)}
    if case["traces"] > 1:
        out = ctx.eval_placements_multi(s["traces"], s["offsets"], s["inst"], case["budget"], flags=case["flags"])
        idx, rec = ctx.topk(out.view(-1, 128), case["k"])
    else:
        out = ctx.eval_placements(s["traces"][0], s["offsets"], s["inst"], case["budget"], class_mask=s.get("mask"),
                                  flags=case["flags"])
        idx, rec = ctx.topk(out, case["k"])
    return {"records": out.view(torch.int64), "idx": idx, "rec": rec.view(torch.int64)}


def work(case):
    """Bytes: the trace(s) (16 per request), the placements (about 4 + 4 per instance), the records and what is
    ranked or written beside them, once each.  Operations: one decision per request and placement."""
    do = case["do"]
    if do == "rank":
        n = case["n_cand"]
        return {"bytes": n * (128 + 256 + 8 + 3 * 8) + 2 * case["k"] * 132, "flops": 0}
    n, t = case["n_req"], case.get("traces", 1)
    if do == "replan":  # the probes of the pruning are the part whose number is known beforehand
        return {"bytes": 16 * n, "flops": len(STRATEGIES) * len(BATCHES) * n}
    c = case["n_cand"]
    insts = {"tiny": 3, "node": 5, "multi": 6, "paper": 6, "large": 80}[case["space"]]
    b = t * n * 16 + c * (4 + 4 * insts) + t * c * 128 + (case.get("k", 0)) * 132
    if do == "inspect":
        b += -(-c // 2) * n * 20 + c * (64 + 256 + 32 + 8)
    return {"bytes": b, "flops": c * n * t}


def tolerance(case):
    """Whole numbers throughout; the scores are IEEE doubles computed in a stated order without fusing."""
    return "exact"
