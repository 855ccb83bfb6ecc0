"""GPU parity of the standalone ranking (victims, TIDE fill, keys) against the
CPU oracle: bit-exact on every output index and key."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

P_Z = 500_000_000
KVB = 131072
GIB = 1 << 30


@pytest.fixture(scope="module")
def B():
    from paper_2609_09643_gb300 import native
    native.build()
    from paper_2609_09643_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def sigma():
    _, s = oracle.hazard_lut(synth.geometric_turns(1, 1415, 23.7, 2, 200))
    return s


def run(B, recs, params, keys=False):
    import torch
    devs = [B.records_to_device(r) for r in recs]
    outs = [B.rank_outputs(r.n, p["k"], p["max_moves"], keys) for r, p in zip(recs, params)]
    B.rank_batch(devs, params, outs)
    torch.cuda.synchronize()
    return [B.rank_result(o) for o in outs]


def check(r, rec, p, keys=False):
    o = oracle.rank(rec, p["sigma_q"], p["penalty_q"], p["k"], p["budget_bytes"], p["kv_bytes_per_token"],
                    p["free_fast_tok"], p["free_hbm_tok"], keys=keys, max_moves=max(p["max_moves"], 1))
    compare(r, o, p, keys)


def compare(r, o, p, keys=False):
    if p["max_moves"] == 0:
        o["promote"] = o["promote"][:0]
        o["demote"] = o["demote"][:0]
        o["moved_bytes"] = 0
    assert r["status"] == 0
    assert np.array_equal(r["victims"], o["victims"]), "victims"
    assert np.array_equal(r["promote"], o["promote"]), ("promote", r["promote"][:8], o["promote"][:8])
    assert np.array_equal(r["demote"], o["demote"]), ("demote", r["demote"][:8], o["demote"][:8])
    assert r["moved_bytes"] == o["moved_bytes"], "moved"
    if keys:
        assert np.array_equal(r["keys"], o["keys"]), "keys"


def prm(sig, k=1024, budget=16 * GIB, max_moves=1024, free_s=0, free_h=1 << 40):
    return dict(sigma_q=sig, k=k, penalty_q=P_Z, budget_bytes=budget, kv_bytes_per_token=KVB, max_moves=max_moves,
                free_fast_tok=free_s, free_hbm_tok=free_h)


def test_sigma_from_device_table(B):
    """The chain the library offers end to end: the survival table built on
    the device from turn counts (unison_hazard_lut, eqs. hazard/hq/survq)
    feeds the ranking call, and the victims and fill equal the oracle's with
    the oracle's own table."""
    import torch
    tps = synth.geometric_turns(2, 5000, 23.7, 2, 200)
    turns = torch.from_numpy(np.asarray(tps, dtype=np.int32)).to("cuda")
    sig_dev, _ = B.hazard_lut(turns)
    sig = sig_dev.cpu().numpy().view(np.uint16)
    _, sig_oracle = oracle.hazard_lut(tps)
    assert np.array_equal(sig, sig_oracle)
    rec = synth.make_records(21, 300_000)
    ps = [prm(sig, k=k, budget=b, free_s=fs) for k, b, fs in [(1024, 8 * GIB, 0), (64, 64 * GIB, 50_000)]]
    res = run(B, [rec] * len(ps), ps)
    for r, p in zip(res, ps):
        o = oracle.rank(rec, sig_oracle, p["penalty_q"], p["k"], p["budget_bytes"], p["kv_bytes_per_token"],
                        p["free_fast_tok"], p["free_hbm_tok"], max_moves=p["max_moves"])
        compare(r, o, p)


@pytest.mark.parametrize("n", [1, 7, 1000, 2047, 2049, 4096, 16384])
def test_small_sets_all_candidates(B, sigma, n):
    rec = synth.make_records(n, n)
    ps = [prm(sigma, k=k, budget=b, free_s=fs) for k, b, fs in
          [(1, 1 * GIB, 0), (5, 64 * GIB, 0), (1024, 4 * GIB, 30000), (4096, 1 << 50, 10 ** 7)]]
    res = run(B, [rec] * len(ps), ps, keys=True)
    for r, p in zip(res, ps):
        check(r, rec, p, keys=True)


@pytest.mark.parametrize("n", [16385, 1 << 17, 1 << 18, 1 << 20])
def test_sampled_sizes(B, sigma, n):
    rec = synth.make_records(11, n)
    ps = [prm(sigma, k=k, budget=b) for k, b in [(1, 1 * GIB), (64, 8 * GIB), (1024, 64 * GIB)]]
    res = run(B, [rec] * len(ps), ps, keys=(n <= (1 << 18)))
    for r, p in zip(res, ps):
        check(r, rec, p, keys=(n <= (1 << 18)))


def test_full_size_2p24(B, sigma):
    """The largest live set (2^24 records): victims, fill and every key."""
    rec = synth.make_records(4, 1 << 24)
    p = prm(sigma, k=1024, budget=64 * GIB)
    r = run(B, [rec], [p], keys=True)[0]
    check(r, rec, p, keys=True)


def test_bench_launch_seven_sets(B, sigma):
    """The benchmark's ranking launch: seven copies of one 2^24-record live
    set with TIDE budgets 1..64 GiB and k = 1,024, in one call.  Every set's
    victims, moves and moved bytes equal the oracle's (a spawn pool runs the
    seven oracle rankings, each worker building the set itself)."""
    import multiprocessing as mp
    from cases import oracle_rank_job
    rec = synth.make_records(4, 1 << 24)
    ps = [prm(sigma, k=1024, budget=b * GIB) for b in (1, 2, 4, 8, 16, 32, 64)]
    res = run(B, [rec] * len(ps), ps)
    with mp.get_context("spawn").Pool(len(ps)) as pool:
        ores = pool.map(oracle_rank_job, [(4, 1 << 24, p) for p in ps], chunksize=1)
    for r, o, p in zip(res, ores, ps):
        compare(r, o, p)


def _sorted_records(n, ascending=True):
    rec = synth.make_records(5, n)
    order = np.argsort(rec.gap_q.astype(np.int64), kind="stable")
    if not ascending:
        order = order[::-1]
    f = lambda a: np.ascontiguousarray(a[order])
    rec2 = synth.Records(f(rec.gap_q), f(rec.last_ret), np.zeros(n, np.uint16), f(rec.kv_tok), f(rec.tier),
                         (f(rec.flags) & 1).astype(np.uint8))
    return rec2


@pytest.mark.parametrize("asc", [True, False])
def test_adversarial_order(B, sigma, asc):
    """Records sorted by key put every top record in one region: the sampled
    thresholds miss and the exact re-selection must still give the answer."""
    rec = _sorted_records(1 << 20, asc)
    ps = [prm(sigma, k=1024, budget=64 * GIB), prm(sigma, k=3000, budget=1 << 50, max_moves=4096)]
    for r, p in zip(run(B, [rec] * 2, ps), ps):
        check(r, rec, p)


def test_massive_ties(B, sigma):
    n = 300000
    rec = synth.make_records(6, n)
    rec = synth.Records(np.zeros(n, np.uint32), rec.last_ret, np.zeros(n, np.uint16), rec.kv_tok, rec.tier,
                        np.zeros(n, np.uint8))
    ps = [prm(sigma, k=777, budget=64 * GIB), prm(sigma, k=4096, budget=1 << 45, free_s=50000, max_moves=4096)]
    for r, p in zip(run(B, [rec] * 2, ps, keys=True), ps):
        check(r, rec, p, keys=True)


def test_crowded_buckets(B, sigma):
    """A few records whose keys sit far above thousands of equal ones: below
    the candidates' common prefix every equal-key record falls in one bucket,
    so the finish's bucket cut keeps them all (the radix select when they
    exceed 4,096) and the bucket sort declines for the sorting network."""
    n = 300000
    base = synth.make_records(11, n)
    gap = np.zeros(n, np.uint32)
    gap[np.arange(0, n, n // 7)[:7]] = 1 << 30  # seven far larger gap averages
    rec = synth.Records(gap, base.last_ret, np.zeros(n, np.uint16), base.kv_tok, base.tier, np.zeros(n, np.uint8))
    ps = [prm(sigma, k=1024, budget=64 * GIB), prm(sigma, k=4096, budget=1 << 45, free_s=50000, max_moves=4096)]
    for r, p in zip(run(B, [rec] * 2, ps), ps):
        check(r, rec, p)


@pytest.mark.parametrize("n", [4096, 4097, 9000, 16385, 70_000])
def test_selection_of_crowded_values(B, sigma, n):
    """Sets on both sides of the largest unsampled one (4,096 records), of
    values that crowd: one gap in a hundred spread over nine octaves, the rest
    below 60 us (many equal, and many of key 0), every seventh completed.  A
    selection then takes several cuts and its sort's buckets are uneven; list
    lengths beside the two sorts' limits (512) and at the most wanted."""
    rng = np.random.default_rng(n)
    gap = np.where(rng.random(n) < 0.01, (2.0 ** rng.uniform(20, 29, n)), rng.integers(0, 60, n)).astype(np.uint32)
    turn = rng.integers(0, 3, n).astype(np.uint16)
    flags = np.where(np.arange(n) % 7 == 0, 2, 0).astype(np.uint8)
    tier = rng.integers(1, 3, n).astype(np.uint8)
    rec = synth.Records(gap, np.zeros(n, np.uint32), turn, rng.integers(1, 3000, n).astype(np.uint32), tier, flags)
    ps = [prm(sigma, k=k, budget=64 * GIB, max_moves=m, free_s=fs)
          for k, m, fs in ((1, 512, 10_000), (512, 513, 0), (513, 4096, 1 << 20), (4096, 1, 1 << 20))]
    for r, p in zip(run(B, [rec] * len(ps), ps), ps):
        check(r, rec, p)


@pytest.mark.parametrize("n", [1, 5, 1023, 1025, 4095, 4096, 4097])
def test_small_sets_with_keys_and_as_shards(B, sigma, n):
    """Sets of up to 4,096 records, whose lists are collected by one CTA each:
    sizes beside a thread's four records and a pass of 1,024, every score
    wanted, lists of none, few and more than the set holds; and the same set as
    three shards, merged."""
    import torch
    rec = synth.make_records(900 + n, n)
    ps = [prm(sigma, k=k, budget=b * GIB, max_moves=m, free_s=fs)
          for k, b, m, fs in ((0, 1, 4096, 9000), (16, 64, 64, 0), (4096, 0, 300, 0), (300, 64, 4096, 1 << 30))]
    for r, p in zip(run(B, [rec] * len(ps), ps, keys=True), ps):
        check(r, rec, p, keys=True)
    dev, p = B.records_to_device(rec), ps[1]
    cuts = sorted({0, n // 48 * 16, n // 24 * 16, n})
    parts = []
    for a, b in zip(cuts, cuts[1:]):
        parts.append(B.rank_cands(p["k"], p["max_moves"]))
        B.rank_shard({k: v[a:b] for k, v in dev.items()}, a, p, parts[-1])
    out = B.rank_outputs(n, p["k"], p["max_moves"])
    B.rank_merge(torch.cat(parts), len(parts), p, out)
    torch.cuda.synchronize()
    check(B.rank_result(out), rec, p)


@pytest.mark.parametrize("n_sets,n_tabs", [(2, 2), (64, 2), (65, 1), (64, 3)])
def test_descriptors_with_the_launch_or_uploaded(B, sigma, n_sets, n_tabs):
    """The most sets and distinct survival tables whose descriptors go with the
    launch (64 and 2), and one more of each, which are uploaded."""
    rng = np.random.default_rng(n_sets)
    sigs = [np.clip(sigma.astype(np.int64) - 37 * j, 41, 4095).astype(np.uint16) for j in range(n_tabs)]
    recs = [synth.make_records(200 + i, int(rng.integers(1, 6000))) for i in range(n_sets)]
    ps = [prm(sigs[i % n_tabs], k=20, budget=4 * GIB, max_moves=30, free_s=5000) for i in range(n_sets)]
    for r, rec, p in zip(run(B, recs, ps), recs, ps):
        check(r, rec, p)


def test_calls_of_changing_size_on_one_stream(B, sigma):
    """Single sets, which bring their descriptor with the launch, and batches,
    sampled and not, growing and shrinking in turn on one stream: each call
    finds its work words and histograms zero whatever the one before it used."""
    import torch
    sizes = [[300], [40_000], [20_000, 500], [50_000], [9000, 9000, 9000, 70_000], [64], [20_000, 500], [120_000], [4097]]
    calls = []
    for j, ns in enumerate(sizes):
        recs = [synth.make_records(70 + 5 * j + i, n) for i, n in enumerate(ns)]
        ps = [prm(sigma, k=100 + 50 * i, budget=8 * GIB, max_moves=200, free_s=5000) for i in range(len(ns))]
        outs = [B.rank_outputs(r.n, p["k"], p["max_moves"]) for r, p in zip(recs, ps)]
        calls.append((recs, ps, outs, B.RankCall([B.records_to_device(r) for r in recs], ps, outs)))
    for _ in range(2):
        for c in calls:
            c[3].run()
    torch.cuda.synchronize()
    for recs, ps, outs, _ in calls:
        for rec, p, o in zip(recs, ps, outs):
            check(B.rank_result(o), rec, p)


def test_degenerate_sets(B, sigma):
    n = 50000
    base = synth.make_records(8, n)
    all_pinned = synth.Records(base.gap_q, base.last_ret, base.turn, base.kv_tok, base.tier,
                               np.ones(n, np.uint8))
    all_fast = synth.Records(base.gap_q, base.last_ret, base.turn, base.kv_tok, np.ones(n, np.uint8), base.flags)
    none_res = synth.Records(base.gap_q, base.last_ret, base.turn, base.kv_tok, np.zeros(n, np.uint8), base.flags)
    cases = [(all_pinned, prm(sigma)), (all_fast, prm(sigma)), (none_res, prm(sigma)),
             (base, prm(sigma, k=0, budget=0, max_moves=0)), (base, prm(sigma, budget=0)),
             (base, prm(sigma, max_moves=3)), (base, prm(sigma, free_h=0)), (base, prm(sigma, budget=1))]
    res = run(B, [c[0] for c in cases], [c[1] for c in cases])
    for r, (rec, p) in zip(res, cases):
        check(r, rec, p)


def test_phase1_promotions(B, sigma):
    rec = synth.make_records(9, 200000)
    ps = [prm(sigma, budget=b, free_s=fs, max_moves=mm) for b, fs, mm in
          [(64 * GIB, 60000, 1024), (1 << 50, 10 ** 6, 4096), (1 << 50, 10 ** 9, 64), (2 * GIB, 10 ** 9, 4096)]]
    for r, p in zip(run(B, [rec] * 4, ps), ps):
        check(r, rec, p)


def test_fill_byte_sums_beyond_2p64(B, sigma):
    """Sizes near 2^32 tokens at 2^24 bytes per token and the largest budget:
    the running byte sums pass 2^64 within a few hundred moves, in phase 1
    (free fast-tier space, random sizes) and in the pair loop (equal sizes,
    one promotion's worth of free space)."""
    n = 100000
    base = synth.make_records(10, n)
    big = synth.rng.randint(11, 0, np.arange(n, dtype=np.uint64), 1 << 31, (1 << 32) - 1).astype(np.uint32)
    rnd = synth.Records(base.gap_q, base.last_ret, base.turn, big, base.tier, base.flags)
    flat = synth.Records(base.gap_q, base.last_ret, base.turn, np.full(n, 0xFFFFFFFF, np.uint32), base.tier,
                         base.flags)
    top = (1 << 64) - 1
    cases = [(rnd, 1 << 62, 1 << 62), (rnd, top, top), (flat, 0xFFFFFFFF, 1 << 62), (flat, 0, top)]
    recs, ps = [], []
    for rec, fs, fh in cases:
        p = prm(sigma, k=64, budget=top, max_moves=4096, free_s=fs, free_h=fh)
        p["kv_bytes_per_token"] = 1 << 24
        recs.append(rec)
        ps.append(p)
    res = run(B, recs, ps)
    for r, rec, p in zip(res, recs, ps):
        check(r, rec, p)
    assert len(res[0]["promote"]) > 100 and len(res[2]["demote"]) > 100


def test_more_sets_than_filter_ctas(B, sigma):
    """600 sampled sets (more than the filter's resident CTAs): every CTA
    deals tiles from all sets instead of owning one set's group."""
    n = 20000
    recs = [synth.make_records(1000 + i, n) for i in range(600)]
    ks = [1, 7, 64, 1024]
    ps = [prm(sigma, k=ks[i % 4], budget=(1 << (i % 7)) * GIB, max_moves=(64, 1024)[i % 2]) for i in range(600)]
    res = run(B, recs, ps)
    for i in list(range(0, 600, 37)) + [599]:
        check(res[i], recs[i], ps[i])


def test_batch_of_mixed_sets(B, sigma):
    recs = [synth.make_records(20 + i, n) for i, n in enumerate([100, 20000, 1 << 18, 3000, 1 << 19])]
    ps = [prm(sigma, k=k, budget=(1 << i) * GIB) for i, k in enumerate([3, 50, 1024, 4096, 700])]
    for r, rec, p in zip(run(B, recs, ps, keys=True), recs, ps):
        check(r, rec, p, keys=True)


@pytest.mark.parametrize("large,small", [(1, 2), (1, 63), (2, 62), (3, 100)])
def test_large_sets_beside_small_ones(B, sigma, large, small):
    """Sets of 2^22 records beside sets of one tile: every small set's CTA is
    one that the large sets' shares must leave, or the groups come to more CTAs
    than are resident at once and the launch is refused."""
    big = synth.make_records(61, 1 << 22)
    recs = [synth.make_records(300 + i, 1000 + 13 * i) for i in range(small)]
    for i in range(large):
        recs.insert(i * small // large, big)
    ps = [prm(sigma, k=40 + i % 3, budget=(1 + i % 5) * GIB, max_moves=50, free_s=5000) for i in range(len(recs))]
    res = run(B, recs, ps)
    whole = [i for i, r in enumerate(recs) if r is big][:1]
    for i in whole + [i for i, r in enumerate(recs) if r is not big]:
        check(res[i], recs[i], ps[i])
    for i, r in enumerate(recs):
        assert res[i]["status"] == 0 and len(res[i]["victims"]) == ps[i]["k"]


def test_keys_exact_at_division_boundaries(B):
    """Every sigma in [41, 4095] (through a table of 51 distinct values per
    run), gaps at multiples of sigma and just below, and the largest gap."""
    import torch
    rs = np.random.default_rng(3)
    for run_i in range(4):
        sig = np.sort(rs.choice(np.arange(41, 4096), size=51, replace=False))[::-1].astype(np.uint16)
        if run_i == 0:
            sig[0], sig[1] = 4095, 41
        gs, ts = [], []
        for t in range(51):
            s = int(sig[t])
            q = rs.integers(0, (2 ** 31 - 1) * 4095 // s, 200)
            for x in np.concatenate([q * s, q * s + s - 1]):
                g = int(x) // 4095
                for dg in (-1, 0, 1):
                    if 0 <= g + dg < 2 ** 31:
                        gs.append(g + dg)
                        ts.append(t)
            gs += [0, 1, 2 ** 31 - 1]
            ts += [t, t, t]
        n = len(gs)
        rec = synth.Records(np.array(gs, np.uint32), np.zeros(n, np.uint32), np.array(ts, np.uint16),
                            np.full(n, 100, np.uint32), np.full(n, 2, np.uint8), np.zeros(n, np.uint8))
        p = dict(sigma_q=sig, k=10, penalty_q=(1 << 32) - 1, budget_bytes=0, kv_bytes_per_token=1, max_moves=0,
                 free_fast_tok=0, free_hbm_tok=0)
        r = run(B, [rec], [p], keys=True)[0]
        o = oracle.rank(rec, sig, p["penalty_q"], 10, 0, 1, 0, 0, keys=True)
        assert np.array_equal(r["keys"], o["keys"])


def test_rank_rejects_bad_args(B, sigma):
    import torch
    rec = synth.make_records(1, 100)
    d = B.records_to_device(rec)
    for bad in (dict(k=5000), dict(max_moves=5000), dict(penalty_q=1 << 32), dict(kv_bytes_per_token=0)):
        p = prm(sigma)
        p.update(bad)
        with pytest.raises(B.UnisonError):
            B.rank_batch([d], [p], [B.rank_outputs(100, 5000, 5000)])
    bad_sig = prm(np.full(51, 40, np.uint16))
    with pytest.raises(B.UnisonError):
        B.rank_batch([d], [bad_sig], [B.rank_outputs(100, 1024, 1024)])
    off = dict(d, gap_q=d["gap_q"][1:])  # misaligned
    with pytest.raises(B.UnisonError):
        B.rank_batch([off], [prm(sigma)], [B.rank_outputs(99, 1024, 1024)])
    empty = {k: v[:0] for k, v in d.items()}  # a live set needs at least one record
    with pytest.raises(B.UnisonError):
        B.rank_batch([empty], [prm(sigma)], [B.rank_outputs(1, 1024, 1024)])


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_random_sets_and_parameters(B, seed):
    """Ten live sets per call with random sizes (1 to 2^20 records), random
    shares of pinned, completed and fast-tier records, gap averages with many
    ties, and random k, move limit, DMA budget, free space, P_Z, KV size and
    hazard table: victims, fill and moved bytes equal the oracle's."""
    rng = np.random.default_rng(1000 + seed)
    recs, ps = [], []
    for j in range(10):
        n = int(rng.choice([1, 3, 100, 2047, 4097, 30000, 200000, 1 << 20]))
        base = synth.make_records(100 * seed + j, n)
        u = rng.random(n)
        p_pin, p_done = rng.choice([0.0, 1 / 64, 0.3]), rng.choice([0.0, 0.05, 0.5])
        flags = np.where(u < p_pin, 1, np.where(u < p_pin + p_done, 2, 0)).astype(np.uint8)
        tier = np.where(rng.random(n) < rng.choice([0.0, 1 / 16, 0.5, 1.0]), 1, 2).astype(np.uint8)
        tier[rng.random(n) < rng.choice([0.0, 0.1])] = 0
        gap = base.gap_q.astype(np.int64)
        if rng.random() < 0.5:  # coarse gaps: many equal keys, ties broken by index
            gap = (gap // 1_000_000) * 1_000_000
        gap = np.clip(gap, 0, (1 << 31) - 1).astype(np.uint32)
        recs.append(synth.Records(gap, base.last_ret, base.turn, base.kv_tok, tier, flags))
        sig = rng.integers(41, 4096, size=51).astype(np.uint16)
        ps.append(dict(sigma_q=sig, k=int(rng.integers(0, 4097)), penalty_q=int(rng.integers(0, 1 << 32)),
                       budget_bytes=int(rng.choice([0, 1 << 30, 1 << 36, 1 << 40, 1 << 44, (1 << 63) + 5])),
                       kv_bytes_per_token=int(rng.choice([1, 1024, 28672, 131072, 1 << 24])),
                       max_moves=int(rng.integers(0, 4097)),
                       free_fast_tok=int(rng.choice([0, 1000, 1 << 20, (1 << 64) - 1])),
                       free_hbm_tok=int(rng.choice([0, 5000, 1 << 40, (1 << 64) - 1]))))
    for r, rec, p in zip(run(B, recs, ps), recs, ps):
        check(r, rec, p)


def test_single_set_entry_point(B, sigma):
    """unison_rank, the one-set form, against the oracle and against the batch
    call on the same set."""
    import torch
    rec = synth.make_records(31, 1 << 20)
    dev = B.records_to_device(rec)
    for p in (prm(sigma), prm(sigma, k=3, budget=2 * GIB, max_moves=64, free_s=20_000)):
        out = B.rank_outputs(rec.n, p["k"], p["max_moves"])
        B.rank(dev, p, out)
        torch.cuda.synchronize()
        r = B.rank_result(out)
        check(r, rec, p)
        (rb,) = run(B, [rec], [p])
        for key in ("victims", "promote", "demote"):
            assert np.array_equal(r[key], rb[key]), key


def test_bounded_waits_report_timeout_and_recover(B, sigma):
    """The test library's short waits: a threshold wait on a flag that nothing
    sets and a tile wait on a barrier that nothing arrives at each run out,
    record UNISON_ERR_TIMEOUT in their set's counts[3] and let the kernel
    finish (the other outputs are still exact).  The next ordinary call on
    the same stream then ranks every set exactly, with status OK."""
    import torch
    from paper_2609_09643_gb300 import native
    native.build_debug()
    D = B.debug_lib()
    recs = [synth.make_records(41 + i, 300_000) for i in range(3)]
    ps = [prm(sigma, k=256, budget=4 * GIB, max_moves=128) for _ in recs]
    devs = [B.records_to_device(r) for r in recs]
    outs = [B.rank_outputs(r.n, p["k"], p["max_moves"]) for r, p in zip(recs, ps)]
    call = B.RankCall(devs, ps, outs, lib_=D)
    stream = torch.cuda.current_stream()
    try:
        assert D.unison_debug_rank_wait_hooks(0, 2) == B.OK
        call.run(stream)
        torch.cuda.synchronize()
        res = [B.rank_result(o) for o in outs]
        assert [r["status"] for r in res] == [B.ERR_TIMEOUT, 0, B.ERR_TIMEOUT]
        for r, rec, p in zip(res, recs, ps):
            r["status"] = 0
            check(r, rec, p)
    finally:
        assert D.unison_debug_rank_wait_hooks(-1, -1) == B.OK
    for o in outs:
        o["counts"].zero_()
    call.run(stream)
    torch.cuda.synchronize()
    for o, rec, p in zip(outs, recs, ps):
        check(B.rank_result(o), rec, p)


def test_older_error_does_not_mislead_ranking_calls(B, sigma):
    """An error that an earlier call left pending is not taken for the launch's:
    each ranking call (batch, shard, merge) reports its own verdict, queues its
    work once and leaves its zero blocks in the state the next call expects."""
    import ctypes
    import torch
    from paper_2609_09643_gb300 import native
    native.build_debug()
    D = B.debug_lib()
    rec, p = synth.make_records(47, 60_000), prm(sigma, k=200, budget=4 * GIB, max_moves=100, free_s=9000)
    dev = B.records_to_device(rec)
    stream = torch.cuda.Stream()
    handle = ctypes.c_void_p(stream.cuda_stream)
    cands = [B.rank_cands(p["k"], p["max_moves"]) for _ in range(2)]
    outs = [B.rank_outputs(rec.n, p["k"], p["max_moves"]) for _ in range(4)]
    torch.cuda.synchronize()
    cp, half = B._rank_params(p), rec.n // 32 * 16
    for o in outs[:2]:  # two calls in a row, then shards and a merge, then one more
        assert D.unison_debug_leave_error() == B.OK
        B.RankCall([dev], [p], [o], lib_=D).run(stream)
    for i, (a, b) in enumerate(((0, half), (half, rec.n))):
        part = B._records({f: v[a:b] for f, v in dev.items()})
        assert D.unison_debug_leave_error() == B.OK
        assert D.unison_rank_shard(ctypes.byref(part), a, ctypes.byref(cp), cands[i].data_ptr(), handle) == B.OK
    stream.synchronize()
    both, mo = torch.cat(cands), B._rank_out(outs[2])
    torch.cuda.synchronize()
    assert D.unison_debug_leave_error() == B.OK
    assert D.unison_rank_merge(both.data_ptr(), 2, ctypes.byref(cp), ctypes.byref(mo), handle) == B.OK
    B.RankCall([dev], [p], [outs[3]], lib_=D).run(stream)
    stream.synchronize()
    for o in outs:
        check(B.rank_result(o), rec, p)


@pytest.mark.parametrize("world", [2, 4])
def test_record_sharded_ranking_equals_whole_set(B, sigma, world):
    """Sec. IV-D's scan split by records: each slice ranked into its candidate
    lists (global indices), the lists gathered (here: concatenated on one
    GPU, as the all-gather lays them out) and merged; the victims, moves and
    moved bytes equal the oracle's for the whole set."""
    import torch
    from paper_2609_09643_gb300 import shard
    n = 1 << 22
    rec = synth.make_records(51, n)
    dev = B.records_to_device(rec)
    for p in (prm(sigma, k=1024, budget=16 * GIB, max_moves=1024),
              prm(sigma, k=37, budget=3 * GIB, max_moves=300, free_s=40_000)):
        parts = []
        for r in range(world):
            off, cnt = shard.record_slice(n, r, world)
            c = B.rank_cands(p["k"], p["max_moves"])
            B.rank_shard({k: v[off:off + cnt] for k, v in dev.items()}, off, p, c)
            parts.append(c)
        out = B.rank_outputs(n, p["k"], p["max_moves"])
        B.rank_merge(torch.cat(parts), world, p, out)
        torch.cuda.synchronize()
        check(B.rank_result(out), rec, p)


def test_captured_calls_replay_beside_ordinary_ones(B, sigma):
    """A single set, a batch and a merge captured into a graph: each replay of
    it ranks exactly, and so do ordinary calls on the stream after the capture
    and between replays (a captured call clears work words of its own)."""
    import torch
    recs = [synth.make_records(81, 3_000), synth.make_records(82, 50_000)]
    ps = [prm(sigma, k=100, budget=GIB, max_moves=64), prm(sigma, k=300, budget=4 * GIB, max_moves=200)]
    devs = [B.records_to_device(r) for r in recs]
    outs = [[B.rank_outputs(r.n, p["k"], p["max_moves"]) for r, p in zip(recs, ps)] for _ in range(2)]
    mout = B.rank_outputs(recs[1].n, ps[1]["k"], ps[1]["max_moves"])
    sout = B.rank_outputs(recs[1].n, ps[1]["k"], ps[1]["max_moves"])
    cands = B.rank_cands(ps[1]["k"], ps[1]["max_moves"])
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    calls = [B.rank_prepare(devs, ps, o) for o in outs]  # the graph's outputs, the ordinary calls'
    single = B.rank_prepare(devs[1:], ps[1:], [sout])
    torch.cuda.synchronize()

    def graphed():
        single.run(stream)
        calls[0].run(stream)
        B.rank_shard(devs[1], 0, ps[1], cands, stream=stream)
        B.rank_merge(cands, 1, ps[1], mout, stream=stream)

    calls[1].run(stream)
    graphed()  # scratch grown before the capture
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        graphed()
    for _ in range(3):
        for o in outs[0] + outs[1] + [mout, sout]:
            o["counts"].zero_()
        torch.cuda.synchronize()
        calls[1].run(stream)
        with torch.cuda.stream(stream):
            graph.replay()
        calls[1].run(stream)
        torch.cuda.synchronize()
        for o in outs:
            for oo, rec, p in zip(o, recs, ps):
                check(B.rank_result(oo), rec, p)
        for oo in (mout, sout):
            check(B.rank_result(oo), recs[1], ps[1])


def _captured_case(B, sigma, n_sets, n_tabs, seed, n=3000):
    """A prepared batch with its records, params and outputs (of sets of up to n
    records), and a function that checks and clears the outputs."""
    import torch
    rng = np.random.default_rng(seed)
    sigs = [np.clip(sigma.astype(np.int64) - 37 * j, 41, 4095).astype(np.uint16) for j in range(n_tabs)]
    recs = [synth.make_records(1000 * seed + i, int(rng.integers(max(1, n // 2), n + 1))) for i in range(n_sets)]
    ps = [prm(sigs[i % n_tabs], k=20 + i % 5, budget=4 * GIB, max_moves=30, free_s=5000) for i in range(n_sets)]
    devs = [B.records_to_device(r) for r in recs]
    outs = [B.rank_outputs(r.n, p["k"], p["max_moves"]) for r, p in zip(recs, ps)]
    torch.cuda.synchronize()

    def verify():
        torch.cuda.synchronize()
        for o, rec, p in zip(outs, recs, ps):
            check(B.rank_result(o), rec, p)
            for name in ("victims", "promote", "demote", "counts", "moved"):
                o[name].zero_()
        torch.cuda.synchronize()

    return B.RankCall(devs, ps, outs), verify


@pytest.mark.parametrize("n_sets,n_tabs", [(1, 1), (2, 2), (65, 1), (5, 3)])
def test_captured_call_shares_nothing_with_ordinary_ones(B, sigma, n_sets, n_tabs):
    """A graph whose descriptors go with its launch or are uploaded, captured as
    the first ranking on its stream: replays of it between ordinary calls that
    upload descriptors, repeat them, grow the stream's scratch and turn the
    staging ring over, and a second graph of the stream, all rank exactly; and
    so do ordinary calls after the graphs are gone."""
    import torch
    stream = torch.cuda.Stream()
    call, verify = _captured_case(B, sigma, n_sets, n_tabs, 3)
    second, verify_second = _captured_case(B, sigma, n_sets, n_tabs, 4, 20_000)
    many, verify_many = _captured_case(B, sigma, 65, 1, 5, 600)
    large, verify_large = _captured_case(B, sigma, 1, 1, 6, 1 << 20)
    graph, graph2 = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        call.run(stream)

    def replay(g):
        with torch.cuda.stream(stream):
            g.replay()

    replay(graph)
    verify()
    many.run(stream)  # uploads its descriptors, which the next call finds there
    replay(graph)
    many.run(stream)
    verify()
    verify_many()
    large.run(stream)  # grows the scratch
    replay(graph)
    many.run(stream)
    with torch.cuda.graph(graph2, stream=stream):
        second.run(stream)
    for i in range(20):  # more uploads than the ring has buffers
        _ring, verify_ring = _captured_case(B, sigma, 65, 1, 7 + i % 2, 50)
        _ring.run(stream)
        verify_ring()
        replay((graph, graph2)[i % 2])
    verify()
    verify_second()
    verify_many()
    verify_large()
    # on two other streams at once, beside ordinary calls
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(s1):
        graph.replay()
    with torch.cuda.stream(s2):
        graph2.replay()
    many.run(stream)
    verify()
    verify_second()
    verify_many()
    del graph, graph2
    torch.cuda.synchronize()
    many.run(stream)
    large.run(stream)
    verify_many()
    verify_large()


def test_captured_shards_and_merge_share_nothing(B, sigma):
    """Shards and their merge captured as the first calls on a stream, replayed
    after an ordinary call that needs more scratch."""
    import torch
    rec, p = synth.make_records(83, 48_000), prm(sigma, k=300, budget=4 * GIB, max_moves=200)
    dev, half = B.records_to_device(rec), 24_000
    out = B.rank_outputs(rec.n, p["k"], p["max_moves"])
    size = B.rank_cands(p["k"], p["max_moves"]).numel()
    both = torch.zeros(2 * size, dtype=torch.uint8, device="cuda")
    large, verify_large = _captured_case(B, sigma, 3, 3, 9, 1 << 20)
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        for i, (a, b) in enumerate(((0, half), (half, rec.n))):
            B.rank_shard({f: v[a:b] for f, v in dev.items()}, a, p, both[i * size:(i + 1) * size], stream=stream)
        B.rank_merge(both, 2, p, out, stream=stream)
    for _ in range(3):
        large.run(stream)
        with torch.cuda.stream(stream):
            graph.replay()
        large.run(stream)
        torch.cuda.synchronize()
        check(B.rank_result(out), rec, p)
        verify_large()
        out["counts"].zero_()


def test_capture_out_of_memory_is_reported(B, sigma):
    """A captured call whose memory cannot be had (an injected failure) returns
    UNISON_ERR_OOM and adds nothing to the graph; the capture goes on."""
    import torch
    call, verify = _captured_case(B, sigma, 2, 1, 11)
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        B.debug_fail_allocations(1)
        with pytest.raises(B.UnisonError) as ei:
            call.run(stream)
        assert ei.value.code == B.ERR_OOM
        call.run(stream)
    with torch.cuda.stream(stream):
        graph.replay()
    verify()


@pytest.mark.parametrize("n", [4_097, 40_001, 1 << 20])
def test_lists_of_unlike_lengths_share_a_sample(B, sigma, n):
    """One sample serves lists of 1 to 4,096 wanted: sets whose shortest list
    is the victims', the moves' or neither, few CTAs a set and many."""
    ks = [(1, 4096), (4096, 1), (64, 1024), (1024, 64), (300, 0), (2, 2)]
    recs = [synth.make_records(90 + i, n) for i in range(2)]
    recs = [recs[i % 2] for i in range(len(ks))]
    ps = [prm(sigma, k=k, budget=16 * GIB, max_moves=m, free_s=10_000) for k, m in ks]
    for r, rec, p in zip(run(B, recs, ps), recs, ps):
        check(r, rec, p)
    for rec, p in zip(recs[:2], ps[:2]):
        check(run(B, [rec], [p])[0], rec, p)
