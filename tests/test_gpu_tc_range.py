"""The digit product on rows and columns of subnormal numbers, through ttm_gemm.

The exact product is formed in integers: a subnormal is an integer times 2^-1074. The bound is that of the
digit product on ordinary operands, 4 K u |A||B| entrywise (u = 2^-53)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (130, 70, 33), (40, 65, 300)])
@pytest.mark.parametrize("which", ["rows of A", "columns of B", "entries of A"])
def test_subnormal_operands(M, N, K, which):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_19747_gb300 as pkg
    pkg.build()
    h = pkg.Handle(0)
    rng = np.random.default_rng(M + N + K)
    # integers times 2^-1074 and integers times 2^960: every product is a normal number
    I = rng.integers(-2 ** 40, 2 ** 40, (M, K))
    J = rng.integers(-2 ** 9, 2 ** 9, (K, N)) * 2 + 1
    I[0, 0] = 12345
    if which == "entries of A":      # mixed with entries just above the smallest normal number
        I[:, ::2] *= 2 ** 14
    ref = I.astype(object) @ J.astype(object)
    A, B = np.ldexp(I.astype(np.float64), -1074), np.ldexp(J.astype(np.float64), 960)
    if which == "columns of B":
        A, B = np.ldexp(J.T.astype(np.float64), 960).copy(), np.ldexp(I.T.astype(np.float64), -1074).copy()
        ref = ref.T
    assert np.any((np.abs(A) < 2.0 ** -1022) & (A != 0)) or np.any((np.abs(B) < 2.0 ** -1022) & (B != 0))
    C = pkg.ttm_gemm(h, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), prec="bf16_split").cpu().numpy()
    ref = np.array([[float(v) for v in row] for row in ref]).reshape(ref.shape) * 2.0 ** -114
    bound = 4 * K * 2.0 ** -53 * (np.abs(I).astype(np.float64) @ np.abs(J).astype(np.float64)) * 2.0 ** -114
    bound = bound.T if which == "columns of B" else bound
    assert np.all(np.abs(C - ref) <= bound)
    h.close()
