"""The bin sort of large results (csrc/k_output.cu) against the CPU oracle, bit for bit.

Sizes: bins of one key to several hundred (a bin holds about 16 keys where the distances spread, all of a
segment's keys where they tie), segments of one bin to thousands, queries without results between them."""
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


@pytest.mark.parametrize("values,d,nq,frac", [
    (256, 24, 60, 1.0),   # every point in range, distances spread: bins of about 16 keys
    (256, 24, 160, 0.3),  # a third of the points, half of the queries without any result
    (2, 16, 60, 1.0),     # at most 17 distances: bins of hundreds of equal distances (the CTA sort)
    (1, 16, 120, 1.0),    # one distance: one bin a segment
])
@pytest.mark.parametrize("relabel", [False, True])
def test_bin_sort_bit_exact(rr, values, d, nq, frac, relabel):
    rng = np.random.default_rng(values * 100 + nq)
    n = 1777
    X = (rng.integers(0, values, size=(n, d)) * (255 // max(1, values - 1))).astype(np.uint8)
    adj, start = rrsynth.build_graph(X, 16, 32, 1.2, seed=5)
    Q = X[rng.choice(n, nq, replace=False)].copy()
    d2 = ((X[None].astype(np.int64) - Q[:, None].astype(np.int64)) ** 2).sum(-1)
    r = np.percentile(d2, 100.0 * frac, axis=1)
    if frac < 1.0:
        r[::2] = -1.0
    gi = rr.Index.from_arrays(X, adj, start)
    oX, oadj, ostart = X, adj, start
    order = np.arange(n)
    if relabel:
        gi.relabel()
        order = _bfs(adj, start)
        new = np.empty(n, np.int64)
        new[order] = np.arange(n)
        oX = X[order]
        oadj = adj[order].astype(np.int64)
        oadj = np.where(oadj < n, new[np.minimum(oadj, n - 1)], 0xFFFFFFFF).astype(np.uint32)
        ostart = int(new[start])
    oi = oracle.Index(oX, oadj, ostart)
    o_ids, o_d, _ = oracle.range_search(oi, Q, r, "greedy", beam=8, threads=os.cpu_count() or 4)
    assert sum(len(x) for x in o_ids) >= 32768  # the library takes the bin sort
    res = gi.range_search(Q, r, "greedy", beam=8)
    for i in range(nq):
        ids, dist = res.query(i)
        assert np.array_equal(ids, order[np.asarray(o_ids[i], np.int64)]), i
        assert np.array_equal(dist.astype(np.int64), np.asarray(o_d[i]).astype(np.int64)), i
    gi.close()


def _bfs(adj, start):
    """Queue order from the start point, rows in slot order, unreached points last."""
    n = len(adj)
    seen = np.zeros(n, bool)
    order = [start]
    seen[start] = True
    for v in order:
        for u in adj[v]:
            if u < n and not seen[u]:
                seen[u] = True
                order.append(int(u))
    return np.concatenate([np.array(order, np.int64), np.nonzero(~seen)[0]])
