"""The bounded waits of the 8-bit exhaustive scan (csrc/k_brute_tc.cu): when a wait's limit runs out, every role leaves,
the call returns RR_EINTERNAL with the guard's code, and the next call on the same index is exact.  With a limit of 0
the first wait of every role gives up; small limits let some tiles through first, or all."""
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


@pytest.mark.parametrize("d,n", [(32, 300), (128, 300_000), (512, 40_000)])
def test_waits_that_run_out(rr, d, n):
    import torch
    rng = np.random.default_rng(d)
    X = rng.integers(0, 256, size=(n, d), dtype=np.uint8)
    Q = X[rng.integers(0, n, 130)].copy()
    gi = rr.Index.from_arrays(X, np.full((n, 2), 0xFFFFFFFF, np.uint32), 0)
    want = gi.brute_force(Q, 100.0)
    assert np.all(np.diff(want.offsets) >= 1)  # each query is a point
    for tries in (0, 1, 2, 5, 20):
        try:
            rr.rr_debug_set("brute_wait_tries", tries)
            try:
                res = gi.brute_force(Q, 100.0)
            except rr.RRError as e:
                assert e.status == rr.RR_EINTERNAL and "code 8" in str(e)
            else:
                assert tries > 0
                assert np.array_equal(res.offsets, want.offsets) and np.array_equal(res.ids, want.ids)
        finally:
            rr.rr_debug_set("brute_wait_tries", -1)
        torch.cuda.synchronize()  # the context is still usable
        res = gi.brute_force(Q, 100.0)
        assert np.array_equal(res.offsets, want.offsets) and np.array_equal(res.ids, want.ids)
    gi.close()
