"""Alg. 2 by a cluster of CTAs per query (csrc/k_bfs.cuh) against the CPU oracle, bit for bit.

Sizes: a bitmap in one CTA, in a pair and in four (indexes of 2 and 4 million points whose graph joins a few
thousand of them), rows of 1, 2 and 4 words a lane with remainders, one query with a
frontier large enough to be handed to the two-pass levels, and a result list that overflows."""
import os

import numpy as np
import pytest

import oracle
import rrsynth

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


def _unique_rows(adj):
    """Repeated entries of a row become padding (a row is the set N_out)."""
    adj = np.sort(adj, axis=1)
    adj[:, 1:][adj[:, 1:] == adj[:, :-1]] = 0xFFFFFFFF
    return adj


def _same(res, o_ids, o_d):
    for i in range(len(o_ids)):
        ids, d = res.query(i)
        assert np.array_equal(ids, o_ids[i]), i
        assert np.array_equal(d.astype(np.int64), np.asarray(o_d[i]).astype(np.int64)), i


@pytest.mark.parametrize("R", [1, 31, 32, 33, 64, 65, 97, 128])
def test_row_widths(rr, R):
    rng = np.random.default_rng(R)
    n, d = 1500, 20
    X = rng.integers(0, 30, size=(n, d), dtype=np.uint8)
    adj = rng.integers(0, n, size=(n, R)).astype(np.uint32)
    adj[rng.random((n, R)) < 0.1] = 0xFFFFFFFF
    adj[:, 0] = (np.arange(n) + 1) % n  # every point is reached
    adj = _unique_rows(adj)
    Q = rng.integers(0, 30, size=(30, d), dtype=np.uint8)
    d2 = ((X[None].astype(np.int64) - Q[:, None].astype(np.int64)) ** 2).sum(-1)
    r = float(np.percentile(d2, 60))
    gi, oi = rr.Index.from_arrays(X, adj, 0), oracle.Index(X, adj, 0)
    for b in (1, 8, 40):
        o_ids, o_d, _ = oracle.range_search(oi, Q, r, "greedy", beam=b, threads=os.cpu_count() or 4)
        _same(gi.range_search(Q, r, "greedy", beam=b), o_ids, o_d)
    gi.close()


def _spread(n, R, m, rng):
    """m points spread over the ids of an n-point index, a random graph on them; the other rows are empty."""
    live = np.sort(rng.choice(n, m, replace=False))
    live[0], live[-1] = 0, n - 1
    adj = np.full((n, R), 0xFFFFFFFF, np.uint32)
    adj[live] = live[rng.integers(0, m, size=(m, R))]
    adj[live, 0] = np.roll(live, -1)
    adj[live] = _unique_rows(adj[live])
    return live, adj


@pytest.mark.parametrize("n,m", [(2_000_000, 3000), (4_000_003, 3000), (1_600_000, 3000)])
def test_bitmaps_over_clusters(rr, n, m):
    """Ids over the whole range, the last one included; every live point in range: all are results."""
    rng = np.random.default_rng(n)
    R, d = 16, 4
    live, adj = _spread(n, R, m, rng)
    X = np.zeros((n, d), np.uint8)
    X[live] = rng.integers(0, 100, size=(m, d))
    Q = rng.integers(0, 100, size=(7, d), dtype=np.uint8)
    gi = rr.Index.from_arrays(X, adj, 0)
    d2 = ((X[live][None].astype(np.int64) - Q[:, None].astype(np.int64)) ** 2).sum(-1)
    res = gi.range_search(Q, float(d2.max()), "greedy", beam=16)
    for i in range(len(Q)):
        o = np.lexsort((live, d2[i]))
        ids, dist = res.query(i)
        assert np.array_equal(ids, live[o]) and np.array_equal(dist, d2[i][o])
    gi.close()


@pytest.mark.parametrize("dtype,n", [("u8", 60_000), ("f32", 60_000), ("u8", 2_000_000)])
def test_hand_over_and_overflow(rr, dtype, n):
    """Few queries that hold every live point: frontiers of tens of thousands go to the two-pass levels, with
    room for the results and, on a fresh index, without (6 * 50,000 results fit the first list, 100 times do not)."""
    rng = np.random.default_rng(3)
    m, R, d = 50_000, 24, 8
    live, adj = _spread(n, R, m, rng)
    X = np.zeros((n, d), np.uint8)
    X[live] = rng.integers(0, 200, size=(m, d))
    if dtype == "f32":
        X = X.astype(np.float32)
    for nq in (6, 100):
        Q = rng.integers(0, 200, size=(nq, d)).astype(X.dtype)
        gi = rr.Index.from_arrays(X, adj, 0)
        d2 = ((X[live][None].astype(np.int64) - Q[:, None].astype(np.int64)) ** 2).sum(-1)
        res = gi.range_search(Q, float(d2.max()), "greedy", beam=16)
        for i in range(nq):
            o = np.lexsort((live, d2[i]))
            ids, dist = res.query(i)
            assert np.array_equal(ids, live[o]) and np.array_equal(dist.astype(np.int64), d2[i][o]), i
        gi.close()
