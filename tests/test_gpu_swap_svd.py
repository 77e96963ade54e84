"""The preconditioned Swap SVD (the default pipeline) on shapes around its block, warp and cluster
limits, wide and tall Swap matrices, rank-deficient and flat spectra, and batches, against the dense
product and the oracle.

Untruncated products match the dense product to 1e-12 (the tolerance of the float64 parity tests);
truncated ones have an error within the oracle's plus 1e-10, and the discarded weight agrees to 1e-8
relative (both sum the same singular values squared, each exact to rounding of the largest)."""

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


def multiply(h, A, B, **kw):
    import paper_2410_19747_gb300 as pkg
    O, rep = pkg.ttm_multiply(h, dev(A), dev(B), **kw)
    return [c.cpu().numpy() for c in O], rep


def relerr(O, P):
    return np.linalg.norm(ott.dense(O) - P) / np.linalg.norm(P)


# (L, d, chi_A, chi_B, cap): Swap matrices up to d cap on a side; the smaller side crosses 16 and 32
# (one block pair), 256 (clusters end), and odd sizes throughout
SHAPES = [(4, 3, 5, 4, 5), (4, 4, 4, 7, 8), (5, 2, 8, 8, 16), (6, 2, 9, 17, 17), (4, 11, 3, 11, 3), (5, 5, 13, 7, 13),
          (4, 16, 16, 16, 16), (4, 17, 16, 15, 16), (4, 31, 9, 33, 11), (3, 40, 41, 17, 29)]


@pytest.mark.parametrize("L,d,ca,cb,cap", SHAPES)
@pytest.mark.parametrize("prec", ["fp64", "bf16_split"])
def test_truncated_like_the_oracle(h, L, d, ca, cb, cap, prec):
    A = ttgen.rand_tt_spectral(L, d, ca, 100 * L + d)
    B = ttgen.rand_tt_spectral(L, d, cb, 100 * L + d + 1)
    P = ott.dense(A) * ott.dense(B)
    for eps in (1e-14, 1e-6):
        O, rep = multiply(h, A, B, eps=eps, chi_max=cap, chi_out=cap, prec=prec)
        Oo, ro = ottm.ttm(A, B, eps=eps, chi_max=cap, chi_out=cap)
        assert ott.bonds_of(O) == ott.bonds_of(Oo)
        assert relerr(O, P) <= relerr(Oo, P) + 1e-10
        assert abs(rep["discarded_weight"] - ro["discarded_weight"]) <= 1e-8 * ro["discarded_weight"] + 1e-28
        assert rep["n_fallback"] == 0 and rep["n_nonconverged"] == 0


# The elimination of G in blocks of four columns: Swap matrices past the largest cluster (smaller side
# above 384), and smaller sides of 4 k + 1, 2, 3 with one, two and several blocks.
@pytest.mark.parametrize("prec", ["fp64", "bf16_split"])
@pytest.mark.parametrize("L,d,ca,cb,cap", [(4, 33, 13, 12, 13), (4, 20, 20, 19, 20), (6, 2, 2, 3, 3), (5, 3, 3, 2, 3),
                                           (4, 5, 3, 5, 3), (4, 7, 5, 3, 5), (4, 11, 5, 4, 5), (4, 23, 9, 7, 9)])
def test_eliminated_in_blocks(h, prec, L, d, ca, cb, cap):
    A = ttgen.rand_tt_spectral(L, d, ca, 300 * L + d)
    B = ttgen.rand_tt_spectral(L, d, cb, 300 * L + d + 1)
    P = ott.dense(A) * ott.dense(B)
    O, rep = multiply(h, A, B, eps=1e-14, chi_max=cap, chi_out=cap, prec=prec)
    Oo, ro = ottm.ttm(A, B, eps=1e-14, chi_max=cap, chi_out=cap)
    assert ott.bonds_of(O) == ott.bonds_of(Oo)
    assert relerr(O, P) <= relerr(Oo, P) + 1e-10
    assert rep["n_fallback"] == 0 and rep["n_nonconverged"] == 0


@pytest.mark.parametrize("L,d,ca,cb", [(4, 4, 4, 3), (7, 2, 6, 5), (4, 9, 7, 5)])
def test_a_small_eps_keeps_the_product(h, L, d, ca, cb):
    A, B = ttgen.rand_tt(L, d, ca, 7), ttgen.rand_tt(L, d, cb, 8)
    O, _ = multiply(h, A, B, eps=1e-26)
    assert relerr(O, ott.dense(A) * ott.dense(B)) <= 1e-12


@pytest.mark.parametrize("L,d,ca,cb,cap", [(5, 2, 3, 4, 0), (4, 6, 5, 7, 0), (4, 3, 4, 4, 27), (3, 33, 20, 33, 0), (5, 2, 4, 4, 7)])
def test_nothing_truncated(h, L, d, ca, cb, cap):
    """eps = 0 without a binding cap takes no SVD: bonds min(m, n) as the oracle's, a right-canonical
    result whose centre carries the norm, nothing discarded. (The last cap binds on some Swaps.)"""
    A, B = ttgen.rand_tt(L, d, ca, 31), ttgen.rand_tt(L, d, cb, 32)
    P = ott.dense(A) * ott.dense(B)
    O, rep = multiply(h, A, B, chi_max=cap)
    Oo, ro = ottm.ttm(A, B, chi_max=cap)
    assert ott.bonds_of(O) == ott.bonds_of(Oo)
    assert relerr(O, P) <= relerr(Oo, P) + 1e-12
    assert abs(rep["norm_out"] - np.linalg.norm(ott.dense(O))) <= 1e-12 * rep["norm_out"]
    for c in O[1:]:
        q = c.reshape(c.shape[0], -1)
        assert np.abs(q @ q.T - np.eye(c.shape[0])).max() <= 1e-12


def test_rank_deficient_trains(h):
    """Bonds that carry a few directions only: most singular values are zero to rounding."""
    rng = np.random.default_rng(5)
    A = ttgen.rand_tt(6, 3, 9, 11)
    B = ttgen.rand_tt(6, 3, 9, 12)
    for T in (A, B):
        for k in range(1, 5):
            u = rng.standard_normal((T[k].shape[0], 2)) @ rng.standard_normal((2, T[k].shape[0]))
            T[k] = np.tensordot(u, T[k], axes=(1, 0))
    P = ott.dense(A) * ott.dense(B)
    for kw in (dict(eps=1e-24), dict(eps=0.0, chi_max=20), dict(eps=1e-24, chi_max=12, chi_out=9)):
        O, rep = multiply(h, A, B, **kw)
        assert relerr(O, P) <= 1e-11, kw
        assert rep["n_nonconverged"] == 0


def test_flat_spectra_and_tiny_norms(h):
    """Degenerate singular values (orthogonal cores, no decay), and a field of norm 1e-60."""
    A = ttgen.rand_tt(8, 2, 16, 21, canon="left")
    B = ttgen.constant_tt(8, 2, 1.0)
    P = ott.dense(A)
    O, _ = multiply(h, A, B, eps=1e-26)
    assert relerr(O, P) <= 1e-12
    O, _ = multiply(h, [A[0] * 1e-60] + A[1:], B, eps=1e-26)
    assert np.linalg.norm(ott.dense(O) * 1e60 - P) <= 1e-12 * np.linalg.norm(P)


def test_batch_beyond_one_group_of_ctas(h):
    import paper_2410_19747_gb300 as pkg
    pairs = [(ttgen.rand_tt_spectral(4, 17, c, 900 + c), ttgen.rand_tt_spectral(4, 17, 20 - c % 7, 950 + c))
             for c in range(6, 21)]
    res, _ = pkg.ttm_multiply_batched(h, [(dev(A), dev(B)) for A, B in pairs], eps=1e-12, chi_max=20)
    for (A, B), O in zip(pairs, res):
        P = ott.dense(A) * ott.dense(B)
        Oo, _ = ottm.ttm(A, B, eps=1e-12, chi_max=20)
        assert relerr([c.cpu().numpy() for c in O], P) <= relerr(Oo, P) + 1e-10


@pytest.mark.parametrize("prec", ["fp64", "bf16_split"])
@pytest.mark.parametrize("d,chi", [(3, 4), (32, 20)])
def test_a_nan_is_reported(h, prec, d, chi):
    import paper_2410_19747_gb300 as pkg
    A, B = ttgen.rand_tt(4, d, chi, 1), ttgen.rand_tt(4, d, chi, 2)
    for bad in (np.nan, np.inf):
        A2 = [c.copy() for c in A]
        A2[2][0, 0, 0] = bad
        with pytest.raises(pkg.TTMError) as e:
            pkg.ttm_multiply(h, dev(A2), dev(B), eps=1e-10, chi_max=chi, prec=prec)
        assert e.value.status == -5
