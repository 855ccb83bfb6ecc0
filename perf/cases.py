"""The workloads this framework is timed on.

Two kinds of work, both through the public binding: batched trace replay
(``replay_batch``, ``replay_batch_async``, ``replay_batch_noalloc``) and the
ranking of live sets (``rank``, ``RankCall``, ``rank_shard`` and
``rank_merge``).  Shapes are those of the repository's tests and benchmark
(tiny, paper-scale, parameter sweep, large pool; live sets of 2^10 to 2^24
records); inputs are drawn from the seed here, with the same distributions.

Every output is a whole number (counters, decision hashes, indices, bytes),
so every case compares exactly.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2609_09643_gb300 import binding as B

GIB = 1 << 30
MIB = 1 << 20

# (weight, median seconds, sigma) of the tool-wait gap mixtures.
MIXES = {"short": ((1.0, 3.0, 1.2),),
         "coding": ((0.7, 1.5, 1.2), (0.3, 30.0, 1.2)),
         "general": ((0.5, 4.0, 1.2), (0.5, 90.0, 1.2))}
POLICIES = ("lru", "timeout", "spear", "spear_tide", "belady", "lru_tide")
KVB = (28672, 131072, 163840)
LUT = 51


def listed():
    paper = dict(kind="replay", sessions=1415, mean_turns=23.7, start_ms=2000.0, persist=0.7)
    return [
        # A quick what-if on one small trace, answered at once: four policies, host results.
        dict(name="replay-tiny", kind="replay", study="policies", entry="batch", sessions=64, mean_turns=12.0,
             start_ms=2000.0, mix="short", persist=0.7, traces=1, replays=4),
        # The main comparison: five policies x two gap mixes x three KV sizes on paper-scale traces.
        dict(paper, name="replay-paper", study="compare", entry="batch", mix="both", traces=2, replays=30),
        # Parameter search: 8 traces x 8 capacity pairs x 16 (window, bucket) settings of SPEAR+TIDE.
        dict(paper, name="replay-sweep", study="sweep", entry="async", mix="coding", traces=8, replays=1024),
        # Online hazard table against the offline table and LRU, with the decision logs that attainment reads.
        dict(paper, name="replay-online", study="online", entry="async", mix="both", traces=2, replays=18),
        # Dual-design ablation: stale snapshots in their three modes, and the live replay of each setting.
        dict(paper, name="replay-stale", study="stale", entry="async", mix="both", traces=2, replays=16),
        # A large pool: tens of thousands of sessions live at once, tiers of hundreds of residents.
        dict(name="replay-pool", kind="replay", study="pool", entry="async", sessions=40000, mean_turns=20.0,
             start_ms=1.0, mix="general", persist=0.7, traces=1, replays=16),
        # One scheduling decision over a small live set.
        dict(name="rank-small", kind="rank", entry="single", sets=1, n=1000, ragged=0, k=16, moves=64, keys=False),
        # One decision over one large live set.
        dict(name="rank-2p20", kind="rank", entry="single", sets=1, n=1 << 20, ragged=0, k=1024, moves=1024,
             keys=False),
        # Many tenants' live sets of odd sizes in one call, with every record's score wanted.
        dict(name="rank-tenants", kind="rank", entry="batch", sets=60, n=16411, ragged=1, k=256, moves=256, keys=True),
        # A fleet of large live sets in one call.
        dict(name="rank-33x2p20", kind="rank", entry="batch", sets=33, n=1 << 20, ragged=0, k=1024, moves=1024,
             keys=False),
        # The largest live sets the call accepts, the benchmark's ranking launch.
        dict(name="rank-7x2p24", kind="rank", entry="batch", sets=7, n=1 << 24, ragged=0, k=1024, moves=1024,
             keys=False),
        # One live set split by records into shards, their candidate lists merged.
        dict(name="rank-shards", kind="rank", entry="shards", sets=4, n=1 << 22, ragged=0, k=1024, moves=1024,
             keys=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(np.log2(lo), np.log2(hi))))


def draw(rng):
    if rng.random() < 0.5:
        study = rng.choice(["policies", "compare", "sweep", "online", "stale", "pool"])
        if study == "pool":
            return dict(kind="replay", study=study, entry="async", sessions=_log_int(rng, 4000, 40000),
                        mean_turns=rng.uniform(6.0, 20.0), start_ms=rng.choice([1.0, 5.0]), mix="general", persist=0.7,
                        traces=1, replays=_log_int(rng, 1, 16))
        most = {"policies": 64, "compare": 64, "sweep": 1024, "online": 24, "stale": 24}[study]
        return dict(kind="replay", study=study,
                    entry=rng.choice(["batch", "async"] + (["noalloc"] if study == "policies" else [])),
                    sessions=_log_int(rng, 24, 600 if study == "policies" else 1415), mean_turns=rng.uniform(4.0, 23.7),
                    start_ms=rng.choice([500.0, 2000.0]), mix=rng.choice(["short", "coding", "general", "both"]),
                    persist=rng.choice([0.0, 0.7]), traces=rng.randint(1, 4), replays=_log_int(rng, 1, most))
    entry = rng.choice(["single", "batch", "batch", "shards"])
    keys = entry != "shards" and rng.random() < 0.25
    k, moves = _log_int(rng, 1, 4096), _log_int(rng, 1, 4096)
    if entry == "single":
        return dict(kind="rank", entry=entry, sets=1, n=_log_int(rng, 1 << 9, 1 << 24), ragged=0, k=k, moves=moves,
                    keys=keys)
    if entry == "shards":
        shards = rng.randint(2, 8)
        return dict(kind="rank", entry=entry, sets=shards, n=_log_int(rng, 1 << 12, (1 << 24) // shards), ragged=0, k=k,
                    moves=moves, keys=False)
    n = _log_int(rng, 1 << 9, 1 << 24)
    sets = max(1, min(_log_int(rng, 1, 64), (6 << 24) // n // (3 if keys else 1)))
    return dict(kind="rank", entry=entry, sets=sets, n=n, ragged=rng.randint(0, 1), k=k, moves=moves, keys=keys)


# ----------------------------------------------------------------- traces --
class _Turns:
    """Turn records of one trace (the fields binding.Trace takes)."""

    def __init__(self, seed, sessions, mean_turns, start_ms, mix, persist):
        r = np.random.default_rng([seed, sessions])
        t_s = np.clip(1 + r.geometric(1.0 / max(mean_turns - 1.0, 1.0), sessions), 2, 200).astype(np.int64)
        off = np.zeros(sessions + 1, np.int64)
        off[1:] = np.cumsum(t_s)
        total = int(off[-1])
        sess = np.repeat(np.arange(sessions), t_s)
        first = np.zeros(total, bool)
        first[off[:-1]] = True
        start = np.cumsum(np.rint(r.exponential(start_ms * 1e3, sessions)).astype(np.int64))
        decode = r.integers(64, 257, total)
        ins = np.maximum(np.rint(400.0 * np.exp(0.8 * r.standard_normal(total))), 1).astype(np.int64)
        ins[first] = 2048
        w = np.array([m[0] for m in MIXES[mix]])
        med = np.array([m[1] for m in MIXES[mix]])
        sig = np.array([m[2] for m in MIXES[mix]])
        # a session's gaps recur: component and characteristic interval per session (persist > 0)
        comp = r.choice(len(w), sessions, p=w / w.sum())[sess] if persist > 0 else r.choice(len(w), total, p=w / w.sum())
        z = np.sqrt(persist) * r.standard_normal(sessions)[sess] + np.sqrt(1.0 - persist) * r.standard_normal(total)
        gap = np.clip(np.rint(med[comp] * np.exp(sig[comp] * z) * 1e6), 1, (1 << 31) - 1).astype(np.int64)

        def within(step):  # running sum inside each session
            c = np.cumsum(step)
            return c - np.concatenate(([0], c))[off[:-1]][sess]

        out = within(ins + decode)
        adv = gap + np.concatenate(([0], 20 * decode[:-1]))
        adv[first] = 0
        arrival = start[sess] + within(adv)
        self.turn_off = off.astype(np.uint64)
        self.arrival_us = arrival.astype(np.uint64)
        self.completion_us = (arrival + 20 * decode).astype(np.uint64)
        self.in_tok = (out - decode).astype(np.uint32)
        self.out_tok = out.astype(np.uint32)


def _params(policy, fast, hbm, kvb, trace, **kw):
    return dict(dict(policy=policy, trace_idx=trace, cap_fast_bytes=fast, cap_hbm_bytes=hbm, kv_bytes_per_token=kvb,
                     t_s_ps_per_tok=kvb // 16, t_h_ps_per_tok=kvb // 4), **kw)


def _settings(case, r):
    """The replays of a study, in its own order, cut to the case's count."""
    traces, got = range(case["traces"]), []
    if case["study"] == "policies":
        for i in range(case["replays"]):
            got.append(_params(("lru", "spear", "spear_tide", "belady")[i % 4], (512 << i // 4 % 2) * MIB,
                               (8 << i // 8 % 2) * GIB, 28672, i % case["traces"]))
    elif case["study"] == "compare":
        for kvb in KVB:
            for t in traces:
                got += [_params(p, 4 * GIB, 64 * GIB, kvb, t) for p in POLICIES[:5]]
    elif case["study"] == "sweep":
        for t in traces:
            got += [_params("spear_tide", cs * GIB, ch * GIB, 131072, t, ema_num=2, ema_den=w + 1, hazard_bucket=b)
                    for cs in (1, 2, 4, 8) for ch in (32, 128) for w in (4, 8, 16, 32) for b in (1, 2, 4, 8)]
        order = r.permutation(len(got)) if case["replays"] < len(got) else range(len(got))
        got = [got[i] for i in order]
    elif case["study"] == "online":
        for kvb in KVB:
            for t in traces:
                got += [_params("spear_tide", 4 * GIB, 64 * GIB, kvb, t, hazard_online=True),
                        _params("spear_tide", 4 * GIB, 64 * GIB, kvb, t), _params("lru", 4 * GIB, 64 * GIB, kvb, t)]
    elif case["study"] == "stale":
        for kvb in (131072, 163840):
            for t in traces:
                got += [_params("spear_tide", 4 * GIB, 64 * GIB, kvb, t, stale_sync=mode, stale_m=8)
                        for mode in ("live", "event", "arrivals", "gap_start")]
    else:  # pool
        for i in range(case["replays"]):
            got.append(_params(("spear_tide", "spear_tide", "lru", "spear")[i % 4], (16, 8)[i // 4 % 2] * GIB,
                               (160, 80)[i // 8 % 2] * GIB, 163840, i % case["traces"]))
    while len(got) < case["replays"]:
        # more points of the same study: other hazard buckets and EMA windows
        w = (4, 8, 16, 32)[len(got) % 4]
        got.append(dict(got[len(got) % max(1, min(len(got), 24))], ema_num=2, ema_den=w + 1,
                        hazard_bucket=1 + len(got) % 5))
    return got[:case["replays"]]


def _mix_of(case, t):
    return ("coding", "general")[t % 2] if case["mix"] == "both" else case["mix"]


def _prepare_replay(case, seed):
    r = np.random.default_rng([seed, 7])
    traces = [B.Trace(_Turns(seed * 64 + t, case["sessions"], case["mean_turns"], case["start_ms"], _mix_of(case, t),
                             case["persist"])).upload() for t in range(case["traces"])]
    params = _settings(case, r)
    n = len(params)
    state = dict(traces=traces, params=params,
                 results=torch.zeros((n, B.result_nbytes(1) // 8), dtype=torch.int64, device="cuda"), log=None, cap=0)
    if case["study"] == "online":  # attainment reads the decisions
        state["cap"] = int(10 * case["sessions"] * case["mean_turns"])  # about five decisions an event
        state["log"] = torch.zeros((n, state["cap"], 2), dtype=torch.int32, device="cuda")
    return state


def _run_replay(case, s):
    if case["entry"] == "batch" and s["log"] is None:
        res, _ = B.replay_batch(s["traces"], s["params"])
        mask = (1 << 64) - 1
        return np.array([[x[f] & mask for f in B.RESULT_FIELDS] + [x["status"] & mask] for x in res],
                        dtype=np.uint64).view(np.int64)
    if case["entry"] == "noalloc":
        B.replay_batch_noalloc(s["traces"], s["params"], s["results"])
    else:
        B.replay_batch_async(s["traces"], s["params"], s["results"], log=s["log"], log_capacity=s["cap"])
    return s["results"] if s["log"] is None else (s["results"], s["log"])


# --------------------------------------------------------------- live sets --
def _records(gen, n):
    """One live set: sessions of the paper-scale coding workload caught at a random moment."""
    u = lambda: torch.rand(n, generator=gen, device="cuda")  # noqa: E731
    t_s = (2 + torch.floor(torch.log1p(-u() * 0.9998) / np.log(1.0 - 1.0 / 23.7))).clamp(2, 200).to(torch.int32)
    t = torch.minimum((u() * t_s).to(torch.int32), t_s - 1)
    pinned = u() < 1.0 / 64.0
    done = ~pinned & (t == t_s - 1)
    z = torch.randn(n, generator=gen, device="cuda")
    gap = (torch.where(u() < 0.7, 1.5, 30.0) * torch.exp(1.2 * z) * 1e6).clamp(1, 2.0e9).to(torch.int32)
    gap[t == 0] = 0
    growth = 545.0 * torch.exp(0.3 * torch.randn(n, generator=gen, device="cuda"))
    kv = 2048 + (t * growth).to(torch.int32) + (64 + u() * 193).to(torch.int32)
    tier = torch.where(u() < 1.0 / 16.0, 1, 2).to(torch.uint8)
    ret = ((1 << 30) + u() * (1 << 30)).to(torch.int64).clamp(max=(1 << 31) - 1).to(torch.int32)
    return dict(gap_q=gap, last_ret=ret, turn=t.to(torch.int16), kv_tok=kv, tier=tier,
                flags=pinned.to(torch.uint8) | (done.to(torch.uint8) << 1))


def _set_sizes(case):
    if not case["ragged"]:
        return [case["n"]] * case["sets"]
    return [max(1, case["n"] * (16 + (7 * i) % 17) // 32 - 3 * i % 11) for i in range(case["sets"])]


def _rank_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    turns = (2 + torch.floor(torch.log1p(-torch.rand(1415, generator=gen, device="cuda") * 0.9998) /
                             np.log(1.0 - 1.0 / 23.7))).clamp(2, 200).to(torch.int32)
    sigma = B.hazard_lut(turns)[0].cpu().numpy().view(np.uint16)
    if case["entry"] == "shards":  # slices of one live set
        n = case["n"] // 16 * 16
        whole = _records(gen, n * case["sets"])
        recs = [{f: v[i * n:(i + 1) * n] for f, v in whole.items()} for i in range(case["sets"])]
    else:
        recs = [_records(gen, n) for n in _set_sizes(case)]
    params = [dict(sigma_q=sigma, k=max(1, case["k"] >> (i % 3)), penalty_q=500_000_000,
                   budget_bytes=(1 << (i % 7)) * GIB, kv_bytes_per_token=131072, max_moves=case["moves"],
                   free_fast_tok=8192 * (i % 4), free_hbm_tok=1 << 40) for i in range(len(recs))]
    return recs, params


def _prepare_rank(case, seed):
    recs, params = _rank_inputs(case, seed)
    n_out = 1 if case["entry"] == "shards" else case["sets"]
    z = lambda m, dt: torch.zeros((n_out, m), dtype=dt, device="cuda")  # noqa: E731
    out = dict(victims=z(case["k"], torch.int32), promote=z(case["moves"], torch.int32),
               demote=z(case["moves"], torch.int32), counts=z(4, torch.int32), moved=z(1, torch.int64))
    sizes = [r["gap_q"].numel() for r in recs]
    if case["keys"]:
        off = np.concatenate(([0], np.cumsum([-(-m // 32) * 32 for m in sizes])))
        out["keys"] = torch.zeros(int(off[-1]), dtype=torch.int64, device="cuda")
    outs = [dict({f: v[i] for f, v in out.items() if f != "keys"},
                 keys=out["keys"][off[i]:off[i] + sizes[i]] if case["keys"] else None) for i in range(n_out)]
    state = dict(recs=recs, params=params, outs=outs, out=out)
    if case["entry"] == "shards":
        p = params[0]
        state["cands"] = [B.rank_cands(p["k"], p["max_moves"]) for _ in recs]
    elif case["entry"] == "batch":
        state["call"] = B.rank_prepare(recs, params, outs)
    return state


def _run_rank(case, s):
    if case["entry"] == "single":
        B.rank(s["recs"][0], s["params"][0], s["outs"][0])
    elif case["entry"] == "batch":
        s["call"].run()
    else:
        off = 0
        for i, rec in enumerate(s["recs"]):
            B.rank_shard(rec, off, s["params"][0], s["cands"][i])
            off += rec["gap_q"].numel()
        # one GPU holds every shard here: the all-gather is a concatenation
        B.rank_merge(torch.cat(s["cands"]), len(s["recs"]), s["params"][0], s["outs"][0])
    return s["out"]


# -------------------------------------------------------------- interface --
def prepare(case, seed):
    s = _prepare_replay(case, seed) if case["kind"] == "replay" else _prepare_rank(case, seed)
    s["case"] = case
    return s


def run(state):
    case = state["case"]
    return _run_replay(case, state) if case["kind"] == "replay" else _run_rank(case, state)


def work(case):
    """Bytes one pass cannot do without.  Replays: every replay reads its
    trace's events once (16 B) with the previous turn's size or the gap average
    and key (12 B), and writes its counters; the rest is a serial chain that
    bytes do not describe.  Ranking: gap, turn, flags and tier of every record
    (8 B), the outputs, and 8 B a record where scores are wanted."""
    if case["kind"] == "replay":
        events = 2.0 * case["sessions"] * case["mean_turns"]
        return {"bytes": case["replays"] * (28.0 * events + B.result_nbytes(1)), "flops": 0.0}
    n = sum(_set_sizes(case))
    lists = (1 if case["entry"] == "shards" else case["sets"]) * 4.0 * (case["k"] + 2 * case["moves"] + 6)
    return {"bytes": (16.0 if case["keys"] else 8.0) * n + lists, "flops": 0.0}


def tolerance(case):
    """Counters, hashes, indices and scores are whole numbers."""
    return "exact"


def exact(case, seed):
    """The ranking's scores and victims in plain 64-bit integers: larger score
    first, then the smaller index, over unpinned resident records.  The fill
    and the replays are chains of integer decisions with no rounding: None."""
    if case["kind"] == "replay":
        return None
    recs, params = _rank_inputs(case, seed)
    if case["entry"] == "shards":
        recs = [{f: torch.cat([r[f] for r in recs]) for f in recs[0]}]
    victims = torch.zeros((len(recs), case["k"]), dtype=torch.int32, device="cuda")
    keys = []
    for i, (r, p) in enumerate(zip(recs, params)):
        sigma = torch.from_numpy(p["sigma_q"].astype(np.int64)).cuda()[r["turn"].long().clamp(max=LUT - 1)]
        key = r["gap_q"].long() * 4095 // sigma + (4095 - sigma) * p["penalty_q"] // 4095
        done = (r["flags"] & 2) != 0  # a completed session ranks above every score
        if case["keys"]:
            score = torch.where(done, -1, key)
            keys += [score, torch.zeros(-key.numel() % 32, dtype=torch.int64, device="cuda")]
        key[done] = (1 << 40) - 1
        at = torch.nonzero(((r["flags"] & 1) == 0) & ((r["tier"] == 1) | (r["tier"] == 2)))[:, 0]
        order = ((key[at] - (1 << 39)) << 24) | (0xFFFFFF - at)
        top = torch.topk(order, min(p["k"], at.numel())).values
        victims[i, :top.numel()] = (0xFFFFFF - (top & 0xFFFFFF)).to(torch.int32)
    got = dict(victims=victims, promote=None, demote=None, counts=None, moved=None)
    return dict(got, keys=torch.cat(keys)) if case["keys"] else got
