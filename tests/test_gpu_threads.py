"""Handles on several host threads: the shared-memory limits of the kernels belong to the function and
the device, so a product of one thread must not lower the limit that another thread's launch needs."""

import threading

import numpy as np
import pytest

import ttgen
from oracle import tt as ott

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (L, d, chi, cap, products): columns of 256 rows in shared memory beside columns of a few
WORK = [(4, 16, 16, 16, 40), (6, 2, 3, 4, 150), (5, 5, 9, 9, 80)]


def test_products_of_different_sizes_on_three_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_19747_gb300 as pkg
    pkg.build()
    errors, start = [], threading.Barrier(len(WORK))

    def multiply(L, d, chi, cap, n):
        try:
            stream = torch.cuda.Stream()
            h = pkg.Handle(0, stream=stream.cuda_stream)
            A, B = ttgen.rand_tt_spectral(L, d, chi, 40 + d), ttgen.rand_tt_spectral(L, d, chi, 50 + d)
            a, b = ([torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in T] for T in (A, B))
            torch.cuda.synchronize()
            ref = None
            start.wait()
            for _ in range(n):
                O, _ = pkg.ttm_multiply(h, a, b, eps=1e-14, chi_max=cap)
                got = [c.cpu().numpy() for c in O]
                ref = ref or got
                # the same launches on the same inputs
                assert ott.diff_norm(got, ref) <= 1e-12 * ott.norm(ref)
            h.close()
        except Exception as e:  # reported by the main thread
            start.abort()
            errors.append("%s, d = %d: %r" % (type(e).__name__, d, e))

    threads = [threading.Thread(target=multiply, args=w) for w in WORK]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
