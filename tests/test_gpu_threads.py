"""Calls on different handles from several threads at once (include/rr.h allows it): batches whose launches of one
kernel take different amounts of shared memory.  The limit of a kernel is shared by the threads, so a launch must not
find it lowered by another thread's smaller one."""
import threading

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


@pytest.mark.parametrize("variant,shapes", [
    ("beam", [(1, 512), (700, 32)]),      # the lookahead CTA: 8 warps and a long beam against 2 and a short one
    ("greedy", [(160, 40), (100, 40)]),   # the expansion: CTAs of 384 and of 768 threads
    ("doubling", [(30, 8), (30, 8)]),     # indexes of different degree
])
def test_launches_of_different_sizes(rr, variant, shapes):
    import torch
    rng = np.random.default_rng(1)
    n, d = 2000, 16
    jobs = []
    for k, (nq, beam) in enumerate(shapes):
        R = (16, 120)[k] if variant == "doubling" else 32
        X = rng.integers(0, 30, size=(n, d), dtype=np.uint8)
        adj = rng.integers(0, n, size=(n, R)).astype(np.uint32)
        adj[:, 0] = (np.arange(n) + 1) % n
        adj = np.sort(adj, axis=1)
        adj[:, 1:][adj[:, 1:] == adj[:, :-1]] = 0xFFFFFFFF
        Q = rng.integers(0, 30, size=(nq, d), dtype=np.uint8)
        r = float(np.percentile(((X[None].astype(int) - Q[:8, None].astype(int)) ** 2).sum(-1), 3))
        gi = rr.Index.from_arrays(X, adj, 0)
        Qd = torch.from_numpy(Q).cuda()
        P = rr.rr_params_init(beam=beam)
        want = gi.range_search(Q, r, variant, beam=beam)
        jobs.append((gi, Qd, r, P, want, torch.cuda.Stream()))
    errors = []

    def work(job):
        gi, Qd, r, P, want, stream = job
        try:
            for _ in range(300):
                _, res = rr.rr_range_search(gi.h, Qd, r, variant, P, stream=stream.cuda_stream)
                total = res.total
                rr.rr_result_free(res)
                assert total == len(want.ids)
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for job in jobs:
        job[0].close()
