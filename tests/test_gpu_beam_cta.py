"""The beam phase with a CTA per query (csrc/k_beam_cta.cu): against the CPU oracle bit for bit over row widths, beams,
ties and the batch sizes at which the number of warps changes, and (fp32, inner product) against the warp form, which
a search with exact counters takes."""
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
    adj[rng.random((n, R)) < 0.1] = 0xFFFFFFFF
    adj[:, 0] = (np.arange(n) + 1) % n  # every point is reached
    adj = np.sort(adj, axis=1)          # repeated entries of a row become padding (a row is a set)
    adj[:, 1:][adj[:, 1:] == adj[:, :-1]] = 0xFFFFFFFF
    return adj


def _check(rr, n, d, R, nq, variants, beams, top=30, dtype=np.uint8, **kw):
    rng = np.random.default_rng(n + R + nq)
    X = rng.integers(0, top, size=(n, d)).astype(dtype)
    adj = _graph(rng, n, R)
    Q = rng.integers(0, top, size=(nq, d)).astype(dtype)
    d2 = ((X[None].astype(np.int64) - Q[:20, None].astype(np.int64)) ** 2).sum(-1)
    r = float(np.percentile(d2, 5))
    gi, oi = rr.Index.from_arrays(X, adj, 0), oracle.Index(X, adj, 0)
    for variant in variants:
        for beam in beams:
            o_ids, o_d, o_st = oracle.range_search(oi, Q, r, variant, beam=beam, threads=os.cpu_count() or 4, **kw)
            res = gi.range_search(Q, r, variant, beam=beam, **kw)
            for i in range(nq):
                ids, dist = res.query(i)
                assert np.array_equal(ids, o_ids[i]), (variant, beam, i)
                assert np.array_equal(dist.astype(np.int64), np.asarray(o_d[i]).astype(np.int64)), (variant, beam, i)
            es = np.array([s["early_stopped"] for s in o_st], bool)
            assert np.array_equal((res.flags & rr.RR_FLAG_EARLY_STOPPED) != 0, es)
    gi.close()


@pytest.mark.parametrize("R", [1, 7, 31, 33, 64, 97, 128])
def test_row_widths(rr, R):
    _check(rr, 2000, 20, R, 10, ("beam", "greedy", "beam_es"), (32, 33, 100, 512))


@pytest.mark.parametrize("nq", [1, 304, 305, 608, 609, 1216, 1217])
def test_batch_sizes(rr, nq):
    _check(rr, 1000, 24, 16, nq, ("beam", "greedy_es"), (40,), dtype=np.int8)


def test_ties(rr):
    """4-valued coordinates: long runs of equal distances, more than a beam holds."""
    _check(rr, 3000, 8, 24, 30, ("beam", "greedy", "beam_es"), (32, 64, 200), top=4)


@pytest.mark.parametrize("d,metric", [(100, "ip"), (200, "l2"), (400, "ip")])
def test_fp32_equals_warp_form(rr, d, metric):
    rng = np.random.default_rng(d)
    n, nq = 3000, 50
    X = rng.standard_normal((n, d)).astype(np.float32)
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    Q = X[rng.integers(0, n, nq)] + 0.02 * rng.standard_normal((nq, d)).astype(np.float32)
    m = rr.RR_IP if metric == "ip" else rr.RR_L2
    gi = rr.Index.from_arrays(X, _graph(rng, n, 20), 0, metric=m)
    r = -0.1 if metric == "ip" else 1.8
    for variant in ("beam", "beam_es"):
        for beam in (32, 120):
            x = gi.range_search(Q, r, variant, beam=beam)
            y = gi.range_search(Q, r, variant, beam=beam, collect_stats=1)
            assert np.array_equal(x.offsets, y.offsets) and np.array_equal(x.flags, y.flags)
            assert np.array_equal(x.ids, y.ids) and np.array_equal(x.dists, y.dists)
    gi.close()
