"""The distributed Householder QR of the gauge moves at its edges: wide and tall carriages, row
counts around multiples of 32 and 128, column counts around multiples of the columns per CTA, and
batches with more products than SMs (one CTA per product).

The product with a constant train only moves gauges on the other train, so the dense result is the
input times the constant; every QR is an orthogonal factorisation with an error of a few M u
(u = 2^-53, M <= 1024 rows), which 1e-12 covers at these lengths."""

import numpy as np
import pytest

import ttgen
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


def train(d, bonds, rng):
    D = [1] + list(bonds) + [1]
    return [rng.standard_normal((D[k], d, D[k + 1])) / np.sqrt(D[k]) for k in range(len(D) - 1)]


@pytest.mark.parametrize("d,bonds", [
    (2, (1, 1)), (3, (5, 2)), (2, (2, 33)), (16, (17, 40)), (16, (16, 130)), (31, (31, 37)), (33, (33, 65)),
    (16, (64, 300)), (64, (64, 129)), (32, (40, 1000)),
])
def test_gauge_moves_are_exact(h, d, bonds):
    import paper_2410_19747_gb300 as pkg
    rng = np.random.default_rng(d + sum(bonds))
    A = train(d, bonds, rng)
    B = ttgen.constant_tt(len(A), d, -1.5)
    O, _ = pkg.ttm_multiply(h, dev(A), dev(B), eps=1e-28)
    ref = -1.5 * ott.dense(A)
    got = ott.dense([c.cpu().numpy() for c in O])
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)


def test_a_zero_column_and_a_zero_train(h):
    import paper_2410_19747_gb300 as pkg
    rng = np.random.default_rng(3)
    A = train(4, (7, 6), rng)
    A[0][:, :, 2] = 0.0
    A[1][:, :, 4] = 0.0
    B = ttgen.constant_tt(3, 4, 2.0)
    O, _ = pkg.ttm_multiply(h, dev(A), dev(B), eps=1e-28)
    ref = 2.0 * ott.dense(A)
    assert np.linalg.norm(ott.dense([c.cpu().numpy() for c in O]) - ref) <= 1e-12 * np.linalg.norm(ref)
    Z = [np.zeros_like(c) for c in A]
    O, _ = pkg.ttm_multiply(h, dev(Z), dev(B))
    assert np.abs(ott.dense([c.cpu().numpy() for c in O])).max() == 0.0


@pytest.mark.parametrize("n", [40, 200])
def test_batches_up_to_one_cta_per_product(h, n):
    import paper_2410_19747_gb300 as pkg
    pairs = ttgen.pair_batch(n, 5, 2, 2, 7, 77)
    res, _ = pkg.ttm_multiply_batched(h, [(dev(A), dev(B)) for A, B in pairs])
    for (A, B), O in zip(pairs, res):
        ref = ott.dense(A) * ott.dense(B)
        assert np.linalg.norm(ott.dense([c.cpu().numpy() for c in O]) - ref) <= 1e-12 * np.linalg.norm(ref)
