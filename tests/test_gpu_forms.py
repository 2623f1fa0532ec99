"""Which form of a phase a call takes (rr_debug_count), and each form against the CPU oracle, bit for bit, at the sizes
where the other one is the library's choice next door."""
import functools
import os

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    import paper_2502_13245_gb300 as rr
    rr.build()
    rr.load_library()
    return rr


def _graph(rng, n, R):
    adj = rng.integers(0, n, size=(n, R)).astype(np.uint32)
    adj[:, 0] = (np.arange(n) + 1) % n  # every point is reached
    adj = np.sort(adj, axis=1)          # repeated entries of a row become padding (a row is a set)
    adj[:, 1:][adj[:, 1:] == adj[:, :-1]] = 0xFFFFFFFF
    return adj


def _data(n, d, R, nq, seed, top=30):
    rng = np.random.default_rng(seed)
    X = rng.integers(0, top, size=(n, d), dtype=np.uint8)
    return X, _graph(rng, n, R), rng.integers(0, top, size=(nq, d), dtype=np.uint8)


def _radius(X, Q, share):
    return float(np.percentile(((X[None].astype(np.int64) - Q[:20, None].astype(np.int64)) ** 2).sum(-1), share))


def _same(res, o_ids, o_d):
    for i in range(len(o_ids)):
        ids, d = res.query(i)
        assert np.array_equal(ids, o_ids[i]), i
        assert np.array_equal(d.astype(np.int64), np.asarray(o_d[i]).astype(np.int64)), i


@pytest.mark.parametrize("variant", ["doubling", "doubling_es", "doubling_warm"])
def test_exact_counters_of_doubling_are_kept_by_the_warp_form(rr, variant):
    """rr_query_stats.evals is what the GPU evaluated; the lookahead evaluates more than its rounds keep."""
    X, adj, Q = _data(1500, 16, 20, 30, 1)
    r = _radius(X, Q, 40)
    gi, oi = rr.Index.from_arrays(X, adj, 0), oracle.Index(X, adj, 0)
    o_ids, o_d, o_st = oracle.range_search(oi, Q, r, variant, beam=8, threads=os.cpu_count() or 4)
    warp, cta = rr.rr_debug_count("round_warp"), rr.rr_debug_count("round_cta")
    res = gi.range_search(Q, r, variant, beam=8, collect_stats=1)
    rounds = int(res.stats["rounds"].max())
    assert rounds > 2 and rr.rr_debug_count("round_cta") == cta and rr.rr_debug_count("round_warp") == warp + rounds
    _same(res, o_ids, o_d)
    for key in ("rounds", "distinct", "visits_beam"):
        assert np.array_equal(res.stats[key], [s[key] for s in o_st])
    assert np.all(res.stats["evals"] >= res.stats["distinct"])
    _same(gi.range_search(Q, r, variant, beam=8), o_ids, o_d)
    assert rr.rr_debug_count("round_cta") > cta
    gi.close()


def test_cap_counts_results_not_list_entries(rr):
    """The cluster expansion's warps reserve the item list in chunks and leave most of a small batch's empty; only
    results count against max_results_total.  At the exact number of results nothing is cut and nothing is redone;
    one less cuts."""
    X, adj, Q = _data(3000, 16, 20, 200, 2)
    r = _radius(X, Q, 10)
    gi, oi = rr.Index.from_arrays(X, adj, 0), oracle.Index(X, adj, 0)
    beam = 8
    o_ids, o_d, _ = oracle.range_search(oi, Q, r, "greedy", beam=beam, threads=os.cpu_count() or 4)
    counts = np.array([len(x) for x in o_ids])
    full = int(counts[counts >= beam].sum())
    assert full > beam * (counts >= beam).sum()
    for cap in (full + 1, full):
        cluster, levels = rr.rr_debug_count("greedy_cluster"), rr.rr_debug_count("greedy_levels")
        res = gi.range_search(Q, r, "greedy", beam=beam, max_results_total=cap)
        assert res.status == rr.RR_OK and not np.any(res.flags & rr.RR_FLAG_TRUNCATED)
        assert rr.rr_debug_count("greedy_cluster") == cluster + 1 and rr.rr_debug_count("greedy_levels") == levels
        _same(res, o_ids, o_d)
    res = gi.range_search(Q, r, "greedy", beam=beam, max_results_total=full - 1)
    assert res.status == rr.RR_EOVERFLOW and len(res.ids) == counts.sum() - 1
    gi.close()


@functools.lru_cache(maxsize=1)
def _all_in_range(n, m, R, nq, seed):
    """m of n points joined by a random graph, a radius that holds all of them: every query's results are all m."""
    rng = np.random.default_rng(seed)
    live = np.sort(rng.choice(n, m, replace=False))
    live[0], live[-1] = 0, n - 1
    adj = np.full((n, R), 0xFFFFFFFF, np.uint32)
    row = live[rng.integers(0, m, size=(m, R))].astype(np.uint32)
    row[:, 0] = np.roll(live, -1)
    row = np.sort(row, axis=1)
    row[:, 1:][row[:, 1:] == row[:, :-1]] = 0xFFFFFFFF
    adj[live] = row
    X = np.zeros((n, 8), np.uint8)
    X[live] = rng.integers(0, 200, size=(m, 8))
    return X, adj, live, rng.integers(0, 200, size=(nq, 8), dtype=np.uint8)


def _check_all(res, X, live, Q):
    for i in range(len(Q)):
        d2 = ((X[live].astype(np.int64) - Q[i].astype(np.int64)) ** 2).sum(-1)
        o = np.lexsort((live, d2))
        ids, d = res.query(i)
        assert np.array_equal(ids, live[o]) and np.array_equal(d.astype(np.int64), d2[o]), i


def test_short_item_list_is_grown_and_the_clusters_run_again(rr):
    """5 M results on a fresh index: the first list is too short; the second run fits, and the next call at once."""
    X, adj, live, Q = _all_in_range(60_000, 50_000, 24, 100, 3)
    gi = rr.Index.from_arrays(X, adj, 0)
    for again in (1, 0):
        before = [rr.rr_debug_count("greedy_" + k) for k in ("again", "levels")]
        res = gi.range_search(Q, 1e9, "greedy", beam=16)
        assert [rr.rr_debug_count("greedy_" + k) for k in ("again", "levels")] == [before[0] + again, before[1]]
        _check_all(res, X, live, Q)
    gi.close()


def test_a_capped_call_does_not_expand_everything_first(rr):
    """Results beyond max_results_total are cut by the level kernels; the clusters stop once the cap is exceeded."""
    X, adj, live, Q = _all_in_range(60_000, 50_000, 24, 100, 4)
    gi = rr.Index.from_arrays(X, adj, 0)

    def phase2_ms(**kw):
        best = 1e9
        for _ in range(5):
            res = gi.range_search(Q, 1e9, "greedy", beam=16, profile=1, **kw)
            best = min(best, rr.rr_last_profile(gi.h).phase2_ms)
        return best, res

    full, res = phase2_ms()
    _check_all(res, X, live, Q)
    levels = rr.rr_debug_count("greedy_levels")
    capped, res = phase2_ms(max_results_total=20_000)
    assert rr.rr_debug_count("greedy_levels") == levels + 5
    assert res.status == rr.RR_EOVERFLOW and len(res.ids) == 20_000
    assert np.all((res.flags & rr.RR_FLAG_TRUNCATED) != 0)
    assert capped < full, (capped, full)  # both forms one after the other took longer than the full expansion
    _check_all(gi.range_search(Q, 1e9, "greedy", beam=16), X, live, Q)
    gi.close()


@pytest.mark.parametrize("dtype", ["u8", "f32"])
@pytest.mark.parametrize("nq", [1, 40])
def test_frontier_that_outgrows_its_list_is_handed_over(rr, dtype, nq):
    """From 16 points by rows of 128 the second level holds most of 400,000 points, above the list's 131,072 entries.
    One such query is finished by the level kernels and nothing is done twice; 40 find no room there and are redone."""
    X, adj, live, Q = _all_in_range(420_000, 400_000, 128, 40, 5)
    Q = Q[:nq]
    if dtype == "f32":
        X, Q = X.astype(np.float32), Q.astype(np.float32)
    gi = rr.Index.from_arrays(X, adj, 0)
    handed, levels = rr.rr_debug_count("greedy_handed"), rr.rr_debug_count("greedy_levels")
    res = gi.range_search(Q, 1e9, "greedy", beam=16)
    assert rr.rr_debug_count("greedy_handed") == handed + (1 if nq == 1 else 0)
    assert rr.rr_debug_count("greedy_levels") == levels + (0 if nq == 1 else 1)
    _check_all(res, X, live, Q)
    gi.close()


def test_scratch_of_the_expansion_is_not_taken_before_a_query_needs_it(rr):
    """400 queries of a 3-megabyte index without a result: the search holds its arena and staging, no more."""
    rng = np.random.default_rng(6)
    n, R = 200_000, 4
    X = rng.integers(0, 200, size=(n, 8), dtype=np.uint8)
    gi = rr.Index.from_arrays(X, _graph(rng, n, R), 0)
    Q = rng.integers(0, 200, size=(400, 8), dtype=np.uint8)
    res = gi.range_search(Q, -1.0, "greedy", beam=16)
    assert len(res.ids) == 0
    assert rr.rr_index_info_get(gi.h).scratch_bytes < 32 << 20
    gi.close()


@pytest.mark.parametrize("dtype,d", [("u8", 16), ("u8", 32), ("i8", 48), ("u8", 64), ("i8", 200), ("u8", 512), ("f32", 24)])
@pytest.mark.parametrize("R", [24, 32, 64, 97, 128])
def test_level_kernels_where_the_clusters_find_no_scratch(rr, dtype, d, R):
    """The expansion's own scratch (frontier lists, hand-over) does not fit: the level kernels take the batch, at every
    split of a vector over lanes, by rows (degrees that are multiples of 32) and by pairs."""
    rng = np.random.default_rng(d + R)
    n, nq = 1500, 40
    X = rng.integers(0, 30, size=(n, d)).astype({"u8": np.uint8, "i8": np.int8, "f32": np.float32}[dtype])
    Q = rng.integers(0, 30, size=(nq, d)).astype(X.dtype)
    d2 = ((X[None].astype(np.int64) - Q[:, None].astype(np.int64)) ** 2).sum(-1)
    r = float(np.percentile(d2, 10))
    adj = _graph(rng, n, R)
    oi = oracle.Index(X, adj, 0)
    o_ids, o_d, _ = oracle.range_search(oi, Q, r, "greedy", beam=8, threads=os.cpu_count() or 4)
    assert sum(len(x) for x in o_ids) > nq * 8
    for nth in (3, 4):  # after the arena and the item list: the frontier lists, then the hand-over buffer
        gi = rr.Index.from_arrays(X, adj, 0)
        levels = rr.rr_debug_count("greedy_levels")
        try:
            rr.rr_debug_set("fail_alloc_after", nth)
            res = gi.range_search(Q, r, "greedy", beam=8)
        finally:
            rr.rr_debug_set("fail_alloc_after", -1)
        assert rr.rr_debug_count("greedy_levels") == levels + 1
        _same(res, o_ids, o_d)
        cluster = rr.rr_debug_count("greedy_cluster")
        _same(gi.range_search(Q, r, "greedy", beam=8), o_ids, o_d)
        assert rr.rr_debug_count("greedy_cluster") == cluster + 1
        gi.close()


@pytest.mark.parametrize("n,form", [(1023, "segment_sort"), (1024, "bin_sort")])
@pytest.mark.parametrize("call", ["greedy", "doubling", "brute"])
def test_the_sort_is_chosen_by_results(rr, n, form, call):
    """8 queries that hold every point: 8,184 and 8,192 results.  Empty entries of the cluster expansion's item list do
    not count."""
    X, adj, Q = _data(n, 8, 16, 8, n)
    gi = rr.Index.from_arrays(X, adj, 0)
    before = rr.rr_debug_count(form)
    res = gi.brute_force(Q, 1e9) if call == "brute" else gi.range_search(Q, 1e9, call, beam=16)
    assert rr.rr_debug_count(form) == before + 1
    _check_all(res, X, np.arange(n), Q)
    gi.close()


def test_steps_of_a_redone_phase(rr):
    """rr_profile.phase2_steps of a capped call counts the levels that made the result, not those before it."""
    X, adj, Q = _data(3000, 16, 20, 60, 8)
    r = _radius(X, Q, 10)
    steps = []
    for nth in (-1, 3):  # the clusters first, then the level kernels; the level kernels only
        gi = rr.Index.from_arrays(X, adj, 0)
        try:
            rr.rr_debug_set("fail_alloc_after", nth)
            res = gi.range_search(Q, r, "greedy", beam=8, max_results_total=1000, profile=1)
        finally:
            rr.rr_debug_set("fail_alloc_after", -1)
        assert res.status == rr.RR_EOVERFLOW
        steps.append(rr.rr_last_profile(gi.h).phase2_steps)
        gi.close()
    assert steps[0] == steps[1] > 0


@pytest.mark.parametrize("dtype", ["u8", "i8"])
@pytest.mark.parametrize("metric", ["l2", "ip"])
@pytest.mark.parametrize("on_device", [False, True])
def test_exhaustive_scan_whose_scratch_does_not_fit(rr, dtype, metric, on_device):
    """Without room for the item list the two passes run, without room for the bins the sort of segments; what fits
    the results and their keys still runs."""
    rng = np.random.default_rng(9)
    n, nq, d = 3000, 40, 100
    X = rng.integers(0, 100, size=(n, d)).astype(np.uint8 if dtype == "u8" else np.int8)
    Q = rng.integers(0, 100, size=(nq, d)).astype(X.dtype)
    x, q = X.astype(np.int64), Q.astype(np.int64)
    D = -(q @ x.T) if metric == "ip" else (q * q).sum(1)[:, None] + (x * x).sum(1)[None] - 2 * (q @ x.T)
    r = float(np.percentile(D, 30))
    assert (D <= r).sum() >= 8192
    adj = np.full((n, 2), 0xFFFFFFFF, np.uint32)
    first = 3 if on_device else 1  # after the arena (and the device result's offsets and flags)
    bins = first + (4 if on_device else 2)  # after the item list (and the ids and distances)
    for nth, form in ((first, "brute_two_pass"), (first + 1, "brute_two_pass"), (bins, "segment_sort"), (-1, "bin_sort")):
        gi = rr.Index.from_arrays(X, adj, 0, metric=rr.RR_IP if metric == "ip" else rr.RR_L2)
        before = rr.rr_debug_count(form)
        try:
            rr.rr_debug_set("fail_alloc_after", nth)
            res = rr.rr_brute_force(gi.h, Q, r, result_on_device=on_device)
        finally:
            rr.rr_debug_set("fail_alloc_after", -1)
        assert rr.rr_debug_count(form) == before + 1, (nth, form)
        if on_device:
            host = rr.rr_result_to_host(res)
            rr.rr_result_free(res)
            res = host
        res = rr.RangeResult(res)
        for i in range(nq):
            ids = np.nonzero(D[i] <= r)[0]
            o = np.lexsort((ids, D[i][ids]))
            g_ids, g_d = res.query(i)
            assert np.array_equal(g_ids, ids[o]) and np.array_equal(g_d, D[i][ids[o]]), (nth, i)
        gi.close()


def _tiled(res, nq, o_ids, o_d):
    for i in range(nq):
        ids, d = res.query(i)
        assert np.array_equal(ids, o_ids[i % len(o_ids)]), i
        assert np.array_equal(d.astype(np.int64), np.asarray(o_d[i % len(o_d)]).astype(np.int64)), i


@pytest.mark.parametrize("kw", [dict(), dict(persistent=1), dict(tile_hint=2, seen_log2=6), dict(tile_hint=8, seen_log2=12),
                                dict(persistent=1, tile_hint=1, seen_log2=5), dict(expand=2), dict(persistent=1, expand=3)])
@pytest.mark.parametrize("variant,beam", [("greedy_es", 32), ("beam", 64), ("beam_es", 129), ("greedy", 200), ("beam", 400)])
def test_warp_form_in_every_launch_shape(rr, kw, variant, beam):
    """More queries than the CTA form takes (1,216), with the padded arrays of long beams (129 and more) and without."""
    X, adj, Q = _data(2000, 12, 40, 130, 10)
    r = _radius(X, Q, 12)
    gi, oi = rr.Index.from_arrays(X, adj, 0), oracle.Index(X, adj, 0)
    o_ids, o_d, _ = oracle.range_search(oi, Q, r, variant, beam=beam, expand=kw.get("expand", 1),
                                        threads=os.cpu_count() or 4)
    before = rr.rr_debug_count("beam_warp")
    res = gi.range_search(np.tile(Q, (10, 1)), r, variant, beam=beam, **kw)
    assert rr.rr_debug_count("beam_warp") == before + 1
    _tiled(res, 1300, o_ids, o_d)
    gi.close()


def _unit(rng, n, d):
    X = rng.standard_normal((n, d)).astype(np.float32)
    return X / np.linalg.norm(X, axis=1, keepdims=True)


@pytest.mark.parametrize("d", [100, 200, 500])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("beam", [100, 150, 500])
def test_warp_form_fp32(rr, d, precision, beam):
    """Float rows of one to four chunks a lane: the exact traversal against the CTA form, the low-precision ones against
    the kernel that keeps exact counters."""
    if precision == 1 and d > 256:
        pytest.skip("BF16 traversal takes d <= 256")
    rng = np.random.default_rng(d + beam)
    X = _unit(rng, 2500, d)
    Q = (X[rng.integers(0, len(X), 130)] + 0.02 * rng.standard_normal((130, d))).astype(np.float32)
    gi = rr.Index.from_arrays(X, _graph(rng, len(X), 24), 0, metric=rr.RR_IP)
    for variant in ("beam", "beam_es"):
        kw = dict(beam=beam, precision=precision)
        before = rr.rr_debug_count("beam_warp")
        got = gi.range_search(np.tile(Q, (10, 1)), -0.1, variant, **kw)
        assert rr.rr_debug_count("beam_warp") == before + 1
        want = gi.range_search(Q, -0.1, variant, collect_stats=1 if precision else 0, **kw)
        assert len(want.ids) > 0
        for i in range(1300):
            for g, w in zip(got.query(i), want.query(i % 130)):
                assert np.array_equal(g, w), i
    gi.close()


@pytest.mark.parametrize("L", [129, 300])
def test_construction_with_long_beams(rr, L):
    import rrsynth
    X = np.random.default_rng(L).integers(0, 100, size=(1200, 16), dtype=np.uint8)
    want, start = rrsynth.build_graph(X, 12, L, 1.2, seed=3)
    got, _ = rr.rr_build_graph(X, 12, L, 1.2, passes=2, seed=3, start=start, metric=rr.RR_L2)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("variant", ["doubling", "doubling_es", "doubling_warm", "doubling_warm_es"])
@pytest.mark.parametrize("kind", ["u8", "u8_counters", "f32", "bf16", "fp8"])
def test_doubling_rounds_by_a_warp_per_query(rr, variant, kind):
    """More active queries than the CTA form takes (608); the same queries in small batches go by CTA."""
    rng = np.random.default_rng(11)
    n, d, nq = 900, 16, 650
    if kind.startswith("u8"):
        X = rng.integers(0, 30, size=(n, d), dtype=np.uint8)
        Q = rng.integers(0, 30, size=(50, d), dtype=np.uint8)
        r, metric = _radius(X, Q, 90), rr.RR_L2
    else:
        X = _unit(rng, n, d)
        Q, r, metric = _unit(rng, 50, d), 0.3, rr.RR_IP
    gi = rr.Index.from_arrays(X, _graph(rng, n, 12), 0, metric=metric)
    kw = dict(beam=8, precision={"bf16": 1, "fp8": 2}.get(kind, 0), es_visit_limit=10**6)
    cta = rr.rr_debug_count("round_cta")
    want = gi.range_search(Q, r, variant, **kw)
    assert rr.rr_debug_count("round_cta") > cta
    warp = rr.rr_debug_count("round_warp")
    got = gi.range_search(np.tile(Q, (13, 1)), r, variant, collect_stats=1 if kind == "u8_counters" else 0, **kw)
    assert rr.rr_debug_count("round_warp") > warp
    assert len(want.ids) > 50 * 8
    for i in range(nq):
        for g, w in zip(got.query(i), want.query(i % 50)):
            assert np.array_equal(g, w), i
    gi.close()


@pytest.mark.parametrize("dtype,beam,nq,form", [
    ("u8", 128, 609, "beam_cta"), ("u8", 128, 1216, "beam_cta"), ("u8", 129, 608, "beam_cta"), ("u8", 129, 609, "beam_warp"),
    ("f32", 256, 1216, "beam_cta"), ("f32", 257, 608, "beam_cta"), ("f32", 257, 609, "beam_warp")])
def test_limits_of_the_cta_form(rr, dtype, beam, nq, form):
    """Two warps a query are the slower form for long beams; either side of each limit against the oracle."""
    X, adj, Q = _data(1500, 12, 32, 64, 12)
    r = _radius(X, Q, 12)
    X, Q = X.astype(np.uint8 if dtype == "u8" else np.float32), Q.astype(np.uint8 if dtype == "u8" else np.float32)
    gi, oi = rr.Index.from_arrays(X, adj, 0), oracle.Index(X, adj, 0)
    o_ids, o_d, _ = oracle.range_search(oi, Q, r, "greedy", beam=beam, threads=os.cpu_count() or 4)
    before = rr.rr_debug_count(form)
    res = gi.range_search(np.tile(Q, (20, 1))[:nq], r, "greedy", beam=beam)
    assert rr.rr_debug_count(form) == before + 1
    _tiled(res, nq, o_ids, o_d)
    gi.close()


@pytest.mark.parametrize("dtype", ["u8", "f32"])
def test_last_large_queries_are_handed_over(rr, dtype):
    """Six queries with 50,000 results each: frontiers of thousands while the rest of the chip is idle go to the level
    kernels, which end the phase."""
    X, adj, live, Q = _all_in_range(60_000, 50_000, 24, 6, 13)
    X, Q = (X, Q) if dtype == "u8" else (X.astype(np.float32), Q.astype(np.float32))
    gi = rr.Index.from_arrays(X, adj, 0)
    before = [rr.rr_debug_count("greedy_" + k) for k in ("handed", "levels")]
    res = gi.range_search(Q, 1e9, "greedy", beam=16)
    assert [rr.rr_debug_count("greedy_" + k) for k in ("handed", "levels")] == [before[0] + 6, before[1]]
    _check_all(res, X, live, Q)
    gi.close()


def test_a_device_without_room_for_the_clusters(rr):
    """An index whose frontier lists are large (1 MB a cluster): without room for the larger item list the smaller one
    serves; without room for the lists or the hand-over the level kernels do, and what was taken is given back."""
    X, adj, live, Q = _all_in_range(200_000, 300, 12, 400, 14)
    for nth, form in ((1, "greedy_cluster"), (2, "greedy_cluster"), (3, "greedy_levels"), (4, "greedy_levels")):
        gi = rr.Index.from_arrays(X, adj, 0)
        before = rr.rr_debug_count(form)
        try:
            rr.rr_debug_set("fail_alloc_after", nth)
            res = gi.range_search(Q, 1e9, "greedy", beam=8)
        finally:
            rr.rr_debug_set("fail_alloc_after", -1)
        assert rr.rr_debug_count(form) == before + 1, nth
        _check_all(res, X, live, Q)
        if form == "greedy_levels":  # no frontier list is held
            assert rr.rr_index_info_get(gi.h).scratch_bytes < 152 << 20
        gi.close()
