"""The allocation-free product at the edge of its array: products whose general workspace fits but not
what the faster kernels add run the general kernels alone, and the limit is the general kernels'.

Tolerances as for the other truncated products: an error against the dense product within the
oracle's plus 1e-10."""

import re

import numpy as np
import pytest

import ttgen
from oracle import tt as ott
from oracle import ttm as ottm
from test_zz_no_alloc import _cores, _dev, _noalloc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LIMIT = 16 << 20   # TTM_NOALLOC_SCRATCH_BYTES


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2410_19747_gb300 as pkg
    pkg.build()
    lib = pkg.load_library()
    h = pkg.Handle(0)
    yield pkg, lib, h
    h.close()


@pytest.mark.parametrize("L,d,chi,prec", [(5, 8, 51, "fp64"), (8, 4, 72, "bf16_split"), (4, 16, 26, "fp64")])
def test_the_general_kernels_alone(env, L, d, chi, prec):
    pkg, lib, h = env
    A, B = ttgen.rand_tt_spectral(L, d, chi, 11), ttgen.rand_tt_spectral(L, d, chi, 12)
    kw = dict(eps=1e-14, chi_max=chi, prec=prec)
    _, rep = pkg.ttm_multiply(h, _dev(A), _dev(B), **kw)
    assert rep["peak_workspace_bytes"] > LIMIT   # the faster kernels do not fit
    P = ott.dense(A) * ott.dense(B)
    Oo, _ = ottm.ttm(A, B, eps=1e-14, chi_max=chi)
    bound = np.linalg.norm(ott.dense(Oo) - P) + 1e-10 * np.linalg.norm(P)
    for _ in range(2):
        st, out, bufs = _noalloc(pkg, lib, A, B, **kw)
        assert st == 0, lib.ttm_last_error().decode()
        got = _cores(out, bufs, d)
        assert ott.bonds_of(got) == ott.bonds_of(Oo)
        assert np.linalg.norm(ott.dense(got) - P) <= bound


@pytest.mark.parametrize("L,d,chi", [(5, 8, 52), (20, 2, 256)])
def test_the_limit_does_not_depend_on_the_pipeline(env, L, d, chi):
    """The workspace that a refusal names is the general pipeline's (f32_passes = 3 asks for it)."""
    pkg, lib, h = env
    A, B = ttgen.rand_tt_spectral(L, d, chi, 11), ttgen.rand_tt_spectral(L, d, chi, 12)
    need = []
    for passes in (0, 3):
        st, _, _ = _noalloc(pkg, lib, A, B, eps=1e-14, chi_max=chi, f32_passes=passes)
        assert st == -4
        need.append(int(re.search(rb"needs (\d+) bytes", lib.ttm_last_error()).group(1)))
    assert need[0] == need[1] > LIMIT
