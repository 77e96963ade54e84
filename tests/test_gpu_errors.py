"""A refused launch is reported by the call that met it and by no later one.

The two-site tensor of a Swap is a batch of d^2 GEMMs, and a grid has at most 65535 of them: d = 300 is
refused by the launch."""

import numpy as np
import pytest

import ttgen
from oracle import tt as ott

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(cores):
    return [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in cores]


@pytest.mark.parametrize("kw", [dict(), dict(prec="bf16_split", split_digits=8)])
def test_a_refused_launch_leaves_no_error_behind(kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_19747_gb300 as pkg
    pkg.build()
    h = pkg.Handle(0)
    A, B = ttgen.rand_tt(2, 300, 3, 1), ttgen.rand_tt(2, 300, 2, 2)
    with pytest.raises(pkg.TTMError) as e:
        pkg.ttm_multiply(h, dev(A), dev(B), **kw)
    assert e.value.status == -6
    x = torch.arange(1000, device="cuda", dtype=torch.float64)   # raises an error that is still pending
    assert float((x * 2).sum()) == 999000.0
    A, B = ttgen.rand_tt(4, 3, 3, 1), ttgen.rand_tt(4, 3, 2, 2)
    O, _ = pkg.ttm_multiply(h, dev(A), dev(B), **kw)
    P = ott.dense(A) * ott.dense(B)
    assert np.linalg.norm(ott.dense([c.cpu().numpy() for c in O]) - P) <= 1e-12 * np.linalg.norm(P)
    h.close()
