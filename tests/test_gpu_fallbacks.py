"""The slower paths behind the default pipeline: the float64 Jacobi of a preconditioned Swap whose Newton
steps do not converge, the grid-barrier QR of carriages with more than 2048 rows, and batches whose
products' CTAs cannot all be resident (general pipeline).

Tolerances: untruncated products 1e-12 against the dense product, truncated ones the oracle's error plus
1e-10."""

import numpy as np
import pytest

import ttgen
from oracle import tt as ott
from oracle import ttm as ottm

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


def dev(cores):
    return [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in cores]


def wide_pair(seed):
    """A left-canonical train times a constant: the right parts of the chain are products of square Gaussian
    matrices, whose singular values span ten decades in no particular order of the columns."""
    return ttgen.rand_tt(12, 2, 64, seed, canon="left"), ttgen.constant_tt(12, 2, 1.0)


@pytest.mark.parametrize("kw", [dict(prec="fp64"), dict(prec="bf16_split"), dict(prec="bf16_split", split_digits=8),
                                dict(prec="fp64", use_graph=1)])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_float64_jacobi_of_a_preconditioned_swap(h, seed, kw):
    import paper_2410_19747_gb300 as pkg
    A, B = wide_pair(seed)
    P = ott.dense(A)
    for _ in range(2):
        O, rep = pkg.ttm_multiply(h, dev(A), dev(B), eps=1e-26, chi_max=64, **kw)
        O = [c.cpu().numpy() for c in O]
        assert rep["jacobi_launches"] == rep["n_swaps"]      # the preconditioned Swap
        assert rep["n_fallback"] > 0 and rep["n_nonconverged"] == 0
        assert np.linalg.norm(ott.dense(O) - P) <= 1e-12 * np.linalg.norm(P)
        for c in O[1:]:
            q = c.reshape(c.shape[0], -1)
            assert np.abs(q @ q.T - np.eye(c.shape[0])).max() <= 1e-12


def test_a_batch_with_and_without_fallbacks(h):
    import paper_2410_19747_gb300 as pkg
    pairs = [wide_pair(0), (ttgen.rand_tt(12, 2, 20, 5), ttgen.rand_tt(12, 2, 3, 6)), wide_pair(1)]
    res, reps = pkg.ttm_multiply_batched(h, [(dev(A), dev(B)) for A, B in pairs], eps=1e-26, chi_max=64)
    assert reps[0]["n_fallback"] > 0 and reps[1]["n_fallback"] == 0 and reps[2]["n_fallback"] > 0
    for i, ((A, B), O) in enumerate(zip(pairs, res)):
        P = ott.dense(A) * ott.dense(B)
        bound = 1e-12 * np.linalg.norm(P)
        if i == 1:   # the cap binds inside the sweep
            Oo, _ = ottm.ttm(A, B, eps=1e-26, chi_max=64)
            bound = np.linalg.norm(ott.dense(Oo) - P) + 1e-10 * np.linalg.norm(P)
        assert np.linalg.norm(ott.dense([c.cpu().numpy() for c in O]) - P) <= bound


@pytest.mark.parametrize("d,bonds", [(40, (60,)), (64, (40, 3))])
def test_gauge_moves_of_more_than_2048_rows(h, d, bonds):
    import paper_2410_19747_gb300 as pkg
    rng = np.random.default_rng(d)
    D = [1] + list(bonds) + [1]
    assert any(d * D[k] > 2048 for k in range(1, len(D) - 1))
    A = [rng.standard_normal((D[k], d, D[k + 1])) / np.sqrt(D[k]) for k in range(len(D) - 1)]
    B = ttgen.constant_tt(len(A), d, -1.5)
    O, _ = pkg.ttm_multiply(h, dev(A), dev(B), eps=1e-28, chi_max=64)
    ref = -1.5 * ott.dense(A)
    assert np.linalg.norm(ott.dense([c.cpu().numpy() for c in O]) - ref) <= 1e-12 * np.linalg.norm(ref)


def test_a_batch_beyond_the_resident_products(h):
    """64 products with Swaps of 256 x 256: 57 fit on the chip at once, so these Swaps take the general
    pipeline (three float32 passes), the smaller ones of the same sweep the preconditioned one."""
    import paper_2410_19747_gb300 as pkg
    pairs = [(ttgen.rand_tt_spectral(4, 16, 16 - s % 3, 700 + s), ttgen.rand_tt_spectral(4, 16, 16 - s % 5, 800 + s)) for s in range(64)]
    kw = dict(eps=1e-14, chi_max=16)
    small, r = pkg.ttm_multiply_batched(h, [(dev(A), dev(B)) for A, B in pairs[:8]], **kw)
    assert r[0]["jacobi_launches"] == r[0]["n_swaps"]
    res, r = pkg.ttm_multiply_batched(h, [(dev(A), dev(B)) for A, B in pairs], **kw)
    assert r[0]["n_swaps"] < r[0]["jacobi_launches"] < 3 * r[0]["n_swaps"]
    for (A, B), O, S in list(zip(pairs, res, small)):
        P = ott.dense(A) * ott.dense(B)
        Oo, _ = ottm.ttm(A, B, **kw)
        for T in (O, S):
            T = [c.cpu().numpy() for c in T]
            assert ott.bonds_of(T) == ott.bonds_of(Oo)
            assert np.linalg.norm(ott.dense(T) - P) <= np.linalg.norm(ott.dense(Oo) - P) + 1e-10 * np.linalg.norm(P)
