"""The float64 GEMM at the edges of its tiles (16 and 32 outputs on a side), K panels (32) and
K splits (2 to 8 CTAs of a cluster), through ttm_gemm against numpy.

A float64 dot product of length K errs by at most K u |a||b| (u = 2^-53) whatever the order of
its sum, and numpy's reference by as much again: the entrywise bound is 2 K u |A||B|."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_19747_gb300 as pkg
    pkg.build()
    hd = pkg.Handle(0)
    yield hd
    hd.close()


@pytest.mark.parametrize("M,N,K", [
    (1, 1, 1), (15, 17, 31), (16, 16, 32), (17, 33, 33), (48, 16, 127), (16, 16, 128), (16, 16, 129),
    (33, 31, 255), (40, 40, 1000), (64, 64, 4097), (5, 700, 260),
    (1120, 1120, 40), (1121, 1105, 33), (1248, 1248, 64),
])
@pytest.mark.parametrize("rows_a,rows_b", [(0, 0), (1, 1)])
def test_entrywise_bound(h, M, N, K, rows_a, rows_b):
    import paper_2410_19747_gb300 as pkg
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    a, b = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    if rows_a:   # column-major operands are passed as they are, row-major ones copied first
        a = a.t().contiguous().t()
    if rows_b:
        b = b.t().contiguous().t()
    C = pkg.ttm_gemm(h, a, b, prec="fp64").cpu().numpy()
    bound = 2 * K * 2.0 ** -53 * (np.abs(A) @ np.abs(B)) + 1e-300
    assert np.all(np.abs(C - A @ B) <= bound)
