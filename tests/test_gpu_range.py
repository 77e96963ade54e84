"""Trains of very small and very large norm: the squares of a carriage's columns leave the normal range
of float64 (norms below 1.5e-154, above 9.5e153) while the columns themselves do not. Swap matrices of at
most 1024 rows throughout.

The scale is a power of two, so the exact result is the unscaled product times it; the tolerances are
those of the same products at norm 1: 1e-12, or for a truncated product the oracle's error plus 1e-10 and
1e-8 of the discarded weight."""

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


def train(d, bonds, seed):
    """Right-canonical, norm 1: the carriages of the preparation sweep have the norm of the train."""
    rng = np.random.default_rng(seed)
    D = [1] + list(bonds) + [1]
    T = [rng.standard_normal((D[k], d, D[k + 1])) for k in range(len(D) - 1)]
    for k in range(len(T) - 1, 0, -1):
        q, r = np.linalg.qr(T[k].reshape(D[k], -1).T)
        T[k] = q.T.reshape(D[k], d, D[k + 1])
        T[k - 1] = np.tensordot(T[k - 1], r.T, axes=(2, 0))
    T[0] /= np.linalg.norm(T[0])
    return T


def scaled(T, e):
    return [np.ldexp(T[0], e)] + T[1:]


def constant(L, d):
    return [np.full((1, d, 1), d ** -0.5) for _ in range(L)]


def check(O, A, B, e):
    ref = ott.dense(A) * ott.dense(B)
    O = [c.cpu().numpy() for c in O]
    O[0] = np.ldexp(O[0], -e)    # the centre: every other core is orthonormal
    assert np.linalg.norm(ott.dense(O) - ref) <= 1e-12 * np.linalg.norm(ref)


# columns in the registers of one warp (at most 128 rows), in shared memory, one CTA and several
SHAPES = [(3, (1, 1)), (3, (3, 2)), (16, (9, 12)), (31, (20, 13)), (130, (1,)), (130, (5,)), (250, (4,)), (255, (2,))]


@pytest.mark.parametrize("e", [-514, -525, -560, -900])
@pytest.mark.parametrize("d,bonds", SHAPES)
def test_gauge_moves_of_a_tiny_train(h, d, bonds, e):
    import paper_2410_19747_gb300 as pkg
    A = train(d, bonds, d + sum(bonds))
    B = constant(len(A), d)
    O, _ = pkg.ttm_multiply(h, dev(scaled(A, e)), dev(B))
    check(O, A, B, e)


@pytest.mark.parametrize("d,L", [(3, 3), (16, 3), (130, 2), (255, 2)])
def test_gauge_moves_of_a_huge_train(h, d, L):
    import paper_2410_19747_gb300 as pkg
    A, B = train(d, (1,) * (L - 1), d), constant(L, d)
    A[0] = np.where(np.arange(d)[None, :, None] == 0, 2.0, A[0])   # a large leading entry
    A[0] *= 0.97 / np.linalg.norm(A[0])
    O, _ = pkg.ttm_multiply(h, dev(scaled(A, 512)), dev(B))
    check(O, A, B, 512)


def test_a_batch_of_tiny_trains(h):
    """More products than CTAs of several columns each: one CTA per product, more than eight columns."""
    import paper_2410_19747_gb300 as pkg
    pairs = [(train(4, (4, 12, 4), s), constant(4, 4)) for s in range(200)]
    exps = [-500 - 2 * s if s % 3 else 0 for s in range(200)]
    res, _ = pkg.ttm_multiply_batched(h, [(dev(scaled(A, e)), dev(B)) for (A, B), e in zip(pairs, exps)])
    for (A, B), e, O in zip(pairs, exps, res):
        check(O, A, B, e)


@pytest.mark.parametrize("prec", [dict(prec="fp64"), dict(prec="bf16_split", split_digits=8)])
@pytest.mark.parametrize("e", [-300, -514, -540, -900, 300, 500])
@pytest.mark.parametrize("L,d,chi,cap", [(5, 3, 5, 6), (4, 16, 16, 16)])
def test_truncated_swaps_of_any_norm(h, L, d, chi, cap, e, prec):
    import paper_2410_19747_gb300 as pkg
    A, B = ttgen.rand_tt_spectral(L, d, chi, 100 * L + d), ttgen.rand_tt_spectral(L, d, chi - 1, 100 * L + d + 1)
    P = ott.dense(A) * ott.dense(B)
    for chi_out in (0, cap - 1):
        Oo, ro = ottm.ttm(A, B, eps=1e-14, chi_max=cap, chi_out=chi_out)
        O, rep = pkg.ttm_multiply(h, dev(scaled(A, e)), dev(B), eps=1e-14, chi_max=cap, chi_out=chi_out, **prec)
        O = [c.cpu().numpy() for c in O]
        c = L - 1 if chi_out else 0    # the centre: the rounding leaves it on the last site
        O[c] = np.ldexp(O[c], -e)
        assert ott.bonds_of(O) == ott.bonds_of(Oo)
        assert np.linalg.norm(ott.dense(O) - P) <= np.linalg.norm(ott.dense(Oo) - P) + 1e-10 * np.linalg.norm(P)
        assert rep["n_fallback"] == 0 and rep["n_nonconverged"] == 0
        if abs(e) <= 400:              # its square is a normal number
            w = np.ldexp(rep["discarded_weight"], -2 * e)
            assert abs(w - ro["discarded_weight"]) <= 1e-8 * ro["discarded_weight"] + 1e-28
