"""The square root and reciprocals of the QR's and the elimination's chains (a float32 seed and one
third-order step) against 80-bit arithmetic, over the exponent range, where the code switches to CUDA's own
square root and division (exponents of 900 and beyond) included.

Bounds, u = 2^-53, from the steps: the seed is good to 2^-20, so the third-order step leaves at most 2^-60 and
the roundings of its last operations count: the square root and the reciprocal of a pivot 4 u, v (one addition
more) 6 u, tau (D = g + |alpha| mu with the error of mu and one rounding, then the reciprocal) 12 u."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_19747_gb300 import _build
    out = str(tmp_path_factory.mktemp("scalars") / "libscalars.so")
    r = subprocess.run([_build._nvcc(), "-std=c++17", "-O3", *_build.ARCH, "-Xcompiler", "-fPIC", "-shared",
                        "-I" + os.path.join(ROOT, "include"), "-I" + _build.CSRC,
                        os.path.join(ROOT, "tests", "c", "scalars.cu"), "-o", out, "-lcudart"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out)


def mantissas(n, e, rng):
    """n numbers of exponent e: random mantissas, the ends of the binade and its float32 neighbours among them."""
    m = 1.0 + rng.random(n)
    m[:6] = [1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -23, 1.0 + 2.0 ** -24, 1.5]
    return np.ldexp(m, e)


EXPONENTS = [0, 1, 2, 3, -1, -2, 17, -38, 127, -126, 128, -150, 500, -501, 897, 898, 899, 900, 901, 902, -897, -898, -899,
             -900, -901, -902, 1000, 1019, -1000, -1021, -1022]


def test_scalars_over_the_exponent_range(lib):
    rng = np.random.default_rng(1)
    g = np.concatenate([mantissas(600, e, rng) for e in EXPONENTS])
    n = g.size
    # leading entries from far below the column's norm up to all of it, of both signs
    alpha = np.sqrt(g) * np.exp2(rng.choice([0.0, 0.0, -1.0, -3.0, -20.0, -60.0], n)) * rng.random(n) * rng.choice([-1.0, 1.0], n)
    alpha[::7] = np.sqrt(g[::7])
    alpha[3::7] = 0.0
    x = [torch.from_numpy(v).cuda() for v in (g, alpha)] + [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(4)]
    torch.cuda.synchronize()
    assert lib.scalars(*[ctypes.c_void_p(t.data_ptr()) for t in x[:2]], n, *[ctypes.c_void_p(t.data_ptr()) for t in x[2:]]) == 0
    beta, vj, tau, inv = [t.cpu().numpy().astype(np.longdouble) for t in x[2:]]
    # 64-bit mantissas; where long double is no wider than that, its own error is far below the bounds
    G, A = g.astype(np.longdouble), np.abs(alpha).astype(np.longdouble)
    mu = np.sqrt(G)
    s = np.where(np.signbit(alpha), -1.0, 1.0)
    assert np.all(np.abs(-s * beta - mu) <= 4 * U * mu)
    assert np.all(np.abs(s * vj - (A + mu)) <= 6 * U * (A + mu))
    D = G + A * mu
    assert np.all(np.abs(tau * D - 1) <= 12 * U)
    assert np.all(np.abs(inv * G - 1) <= 4 * U)


def test_pivots_that_do_not_count(lib):
    """Zero, negative, infinite and NaN pivots have the reciprocal 0; a zero column has tau = 0, a NaN travels on."""
    g = np.array([0.0, -1.0, np.inf, np.nan])
    a = np.array([0.0, 0.0, 1.0, 1.0])
    x = [torch.from_numpy(v).cuda() for v in (g, a)] + [torch.empty(4, dtype=torch.float64, device="cuda") for _ in range(4)]
    torch.cuda.synchronize()
    assert lib.scalars(*[ctypes.c_void_p(t.data_ptr()) for t in x[:2]], 4, *[ctypes.c_void_p(t.data_ptr()) for t in x[2:]]) == 0
    beta, vj, tau, inv = [t.cpu().numpy() for t in x[2:]]
    assert np.all(inv == 0.0)
    assert tau[0] == 0.0 and vj[0] == 0.0 and beta[0] == 0.0
    assert not np.isfinite(beta[2]) and np.isnan(beta[3])
