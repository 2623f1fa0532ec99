"""Alg. 3 with a CTA per query (csrc/k_doubling.cu) against the CPU oracle, bit for bit: row widths that are no
multiple of a warp's part, beams from 1 up, many distance ties, results that end inside and beyond the insertion
buffer, the early stop, the warm restart, and one active query more than the CTA form takes."""
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


def _data(n, d, R, nq, seed, top=30):
    rng = np.random.default_rng(seed)
    X = rng.integers(0, top, size=(n, d), dtype=np.uint8)
    adj = rng.integers(0, n, size=(n, R)).astype(np.uint32)
    adj[rng.random((n, R)) < 0.1] = 0xFFFFFFFF
    adj[:, 0] = (np.arange(n) + 1) % n  # every point is reached
    adj = np.sort(adj, axis=1)          # repeated entries of a row become padding (a row is a set)
    adj[:, 1:][adj[:, 1:] == adj[:, :-1]] = 0xFFFFFFFF
    return X, adj, rng.integers(0, top, size=(nq, d), dtype=np.uint8)


def _check(rr, X, adj, Q, share, variant, beam, **kw):
    d2 = ((X[None].astype(np.int64) - Q[:50, None].astype(np.int64)) ** 2).sum(-1)
    r = float(np.percentile(d2, share))
    gi, oi = rr.Index.from_arrays(X, adj, 0), oracle.Index(X, adj, 0)
    o_ids, o_d, _ = oracle.range_search(oi, Q, r, variant, beam=beam, threads=os.cpu_count() or 4, **kw)
    res = gi.range_search(Q, r, variant, beam=beam, **kw)
    for i in range(len(Q)):
        ids, d = res.query(i)
        assert np.array_equal(ids, o_ids[i]), i
        assert np.array_equal(d.astype(np.int64), np.asarray(o_d[i]).astype(np.int64)), i
    gi.close()


@pytest.mark.parametrize("R", [1, 7, 8, 31, 33, 64, 97, 128])
@pytest.mark.parametrize("variant,beam", [("doubling", 1), ("doubling", 8), ("doubling_es", 20), ("doubling_warm", 8)])
def test_row_widths(rr, R, variant, beam):
    _check(rr, *_data(1500, 20, R, 20, R), 60, variant, beam)


@pytest.mark.parametrize("variant", ["doubling", "doubling_warm"])
def test_ties_and_flushes(rr, variant):
    """4-valued coordinates: whole shells of equal distances; 90% of 6,000 points match."""
    _check(rr, *_data(6000, 8, 16, 12, 5, top=4), 90, variant, 16)


@pytest.mark.parametrize("nq", [608, 609])
def test_form_limit(rr, nq):
    _check(rr, *_data(700, 16, 12, nq, 9), 100, "doubling", 8)
