"""Report fields against what the call did: the largest bond against the chain's trace, the Jacobi launches."""

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


def largest(rep, A, B):
    """A bond of the trains is an input's, or one that a Swap made and that the chain still has at the next
    Contract (a QR makes none above the one it replaces)."""
    return max(rep["bond_trace"] + ott.bonds_of(A) + ott.bonds_of(B))


@pytest.mark.parametrize("kw", [dict(), dict(eps=1e-14, chi_max=6), dict(eps=1e-10, chi_max=12, chi_out=5),
                                dict(chi_max=6, prec="bf16_split"), dict(eps=1e-14, chi_max=6, f32_passes=3),
                                dict(eps=1e-14, chi_max=6, use_graph=1)])
def test_max_bond(h, kw):
    import paper_2410_19747_gb300 as pkg
    A, B = ttgen.rand_tt(7, 3, 6, 61), ttgen.rand_tt(7, 3, 4, 62)
    for _ in range(2):
        _, rep = pkg.ttm_multiply(h, dev(A), dev(B), **kw)
        assert rep["max_bond"] == largest(rep, A, B)
        if kw.get("chi_max"):
            assert rep["max_bond"] <= max(kw["chi_max"], 6)
    pairs = [(A, B), (ttgen.rand_tt(7, 3, 2, 63), ttgen.rand_tt(7, 3, 3, 64))]
    _, reps = pkg.ttm_multiply_batched(h, [(dev(a), dev(b)) for a, b in pairs], **kw)
    for (a, b), rep in zip(pairs, reps):
        assert rep["max_bond"] == largest(rep, a, b)


@pytest.mark.parametrize("kw,per_svd", [(dict(), 0), (dict(eps=1e-14, chi_max=6), 1), (dict(eps=1e-14, chi_max=12, chi_out=5), 1),
                                        (dict(chi_max=6, f32_passes=2), 2), (dict(eps=1e-14, newton_steps=4), 3),
                                        (dict(eps=1e-14, chi_max=6, use_graph=1), 1)])
def test_jacobi_launches(h, kw, per_svd):
    """Float32 Jacobi launches: none where nothing is truncated, one per preconditioned SVD, the passes of
    the general pipeline."""
    import paper_2410_19747_gb300 as pkg
    A, B = ttgen.rand_tt(7, 3, 6, 61), ttgen.rand_tt(7, 3, 4, 62)
    for _ in range(2):
        _, rep = pkg.ttm_multiply(h, dev(A), dev(B), **kw)
        svds = rep["n_swaps"] + (6 if kw.get("chi_out") else 0)
        assert rep["jacobi_launches"] == per_svd * svds
