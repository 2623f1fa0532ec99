"""The warp form of the beam phase with long beams (padded search and shift by source, csrc/k_beam.cu) against the CPU
oracle, bit for bit: beams around the limits of its arrays, rows that bring more and fewer than 32 new keys a visit."""
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


@pytest.mark.parametrize("beam", [128, 129, 255, 256, 257, 511, 512])
@pytest.mark.parametrize("R,top", [(5, 30), (40, 30), (128, 30), (64, 4)])
def test_long_beams(rr, beam, R, top):
    rng = np.random.default_rng(beam + R)
    n, d, nq = 2500, 12, 12
    X = rng.integers(0, top, size=(n, d), dtype=np.uint8)
    adj = rng.integers(0, n, size=(n, R)).astype(np.uint32)
    adj[:, 0] = (np.arange(n) + 1) % n  # every point is reached
    adj = np.sort(adj, axis=1)          # repeated entries of a row become padding (a row is a set)
    adj[:, 1:][adj[:, 1:] == adj[:, :-1]] = 0xFFFFFFFF
    Q = rng.integers(0, top, size=(nq, d), dtype=np.uint8)
    d2 = ((X[None].astype(np.int64) - Q[:, None].astype(np.int64)) ** 2).sum(-1)
    r = float(np.percentile(d2, 8))
    gi, oi = rr.Index.from_arrays(X, adj, 0), oracle.Index(X, adj, 0)
    for variant in ("beam", "beam_es"):
        o_ids, o_d, o_st = oracle.range_search(oi, Q, r, variant, beam=beam, threads=os.cpu_count() or 4)
        res = gi.range_search(Q, r, variant, beam=beam, collect_stats=1)  # exact counters: the warp form
        for i in range(nq):
            ids, dist = res.query(i)
            assert np.array_equal(ids, o_ids[i]), (variant, i)
            assert np.array_equal(dist.astype(np.int64), np.asarray(o_d[i]).astype(np.int64)), (variant, i)
        assert np.array_equal(res.stats["visits_beam"], [s["visits_beam"] for s in o_st])
    gi.close()
