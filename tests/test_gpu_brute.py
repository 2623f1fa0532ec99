"""Exhaustive search (csrc/k_brute_tc.cu) against numpy integers: equal ids, order and distances.

Sizes: row widths on both sides of every tile width of the points, batches around the query tile of 128, point
counts around the tiles, extreme values (the largest sums), radii that match nothing, a few and everything."""
import numpy as np
import pytest

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


def _check(rr, X, Q, metric, radii):
    adj = np.full((len(X), 2), 0xFFFFFFFF, np.uint32)
    gi = rr.Index.from_arrays(X, adj, 0, metric=rr.RR_IP if metric == "ip" else rr.RR_L2)
    x, q = X.astype(np.int64), Q.astype(np.int64)
    D = -(q @ x.T) if metric == "ip" else (q * q).sum(1)[:, None] + (x * x).sum(1)[None] - 2 * (q @ x.T)
    for frac in radii:
        r = np.full(len(Q), float(D.min() - 1)) if frac < 0 else np.floor(np.percentile(D, 100 * frac, axis=1))
        r[1::3] += 1  # radii differ between queries
        res = gi.brute_force(Q, r)
        for i in range(len(Q)):
            ids = np.nonzero(D[i] <= r[i])[0]
            o = np.lexsort((ids, D[i][ids]))
            g_ids, g_d = res.query(i)
            assert np.array_equal(g_ids, ids[o]), (frac, i)
            assert np.array_equal(g_d, D[i][ids[o]]), (frac, i)
    gi.close()


@pytest.mark.parametrize("dtype", ["u8", "i8"])
@pytest.mark.parametrize("metric", ["l2", "ip"])
@pytest.mark.parametrize("d", [1, 16, 63, 64, 65, 100, 128, 129, 192, 256, 257, 320, 384, 400, 449, 512])
def test_row_widths(rr, dtype, metric, d):
    rng = np.random.default_rng(d)
    lo, hi = (0, 256) if dtype == "u8" else (-128, 128)
    t = np.uint8 if dtype == "u8" else np.int8
    _check(rr, rng.integers(lo, hi, size=(1100, d)).astype(t), rng.integers(lo, hi, size=(37, d)).astype(t), metric,
           (-1, 0.0, 0.01, 1.0))


@pytest.mark.parametrize("nq", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("n", [1, 31, 128, 257, 40_000])
def test_ragged_sizes(rr, n, nq):
    rng = np.random.default_rng(n + nq)
    _check(rr, rng.integers(0, 256, size=(n, 96), dtype=np.uint8), rng.integers(0, 256, size=(nq, 96), dtype=np.uint8),
           "l2", (0.0, 0.02))


@pytest.mark.parametrize("dtype", ["u8", "i8"])
@pytest.mark.parametrize("metric", ["l2", "ip"])
@pytest.mark.parametrize("d", [256, 512])
def test_extreme_values(rr, dtype, metric, d):
    """Vectors of the smallest and the largest value only: the largest sums the accumulators meet, and near them
    single steps apart."""
    rng = np.random.default_rng(1)
    lo, hi = (0, 255) if dtype == "u8" else (-128, 127)
    t = np.uint8 if dtype == "u8" else np.int8
    X = np.where(rng.random((600, d)) < np.linspace(0, 1, 600)[:, None], lo, hi).astype(np.int64)
    X[::7, 3] = hi - 1
    Q = np.stack([np.full(d, lo), np.full(d, hi), np.where(np.arange(d) % 2, lo, hi)])
    _check(rr, X.astype(t), Q.astype(t), metric, (0.0, 0.5, 1.0))


def test_list_growth(rr):
    """More matches than the first item list holds (2^20): the pass is repeated with a larger one."""
    rng = np.random.default_rng(2)
    _check(rr, rng.integers(0, 256, size=(9000, 32), dtype=np.uint8), rng.integers(0, 256, size=(160, 32), dtype=np.uint8),
           "l2", (1.0,))
