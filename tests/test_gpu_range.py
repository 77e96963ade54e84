"""Trains of very small and very large norm: the squares of a carriage's columns leave the normal range
of float64 (norms below 1.5e-154, above 9.5e153) while the columns themselves do not. Swap matrices of at
most 1024 rows throughout.

The scale is a power of two, so the exact result is the unscaled product times it; the tolerance is
that of the same products at norm 1 (1e-12)."""

import numpy as np
import pytest

from oracle import tt as ott

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
SHAPES = [(3, (1, 1)), (3, (3, 2)), (16, (9, 12)), (31, (20, 13)), (130, (1,)), (130, (5,)), (250, (40,)), (255, (2,))]


@pytest.mark.parametrize("e", [-514, -525])
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
    exps = [-500 - s % 30 if s % 3 else 0 for s in range(200)]
    res, _ = pkg.ttm_multiply_batched(h, [(dev(scaled(A, e)), dev(B)) for (A, B), e in zip(pairs, exps)])
    for (A, B), e, O in zip(pairs, exps, res):
        check(O, A, B, e)
