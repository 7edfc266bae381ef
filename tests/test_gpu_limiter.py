"""The FP64 van Leer limiter of the sweeps with upwind owners by itself: against the
one with CUDA's divide, and against exact rational arithmetic."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2208_09132_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def limiter(tmp_path_factory):
    import torch
    so = tmp_path_factory.mktemp("limiter") / "limiter_check.so"
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-o", str(so),
                    os.path.join(here, "limiter_check.cu")], check=True, capture_output=True)
    fn = ctypes.CDLL(str(so)).limiter_f64

    def run(s1, s2):
        d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (s1, s2)]
        o = [torch.empty_like(d[0]) for _ in range(2)]
        assert fn(*(ctypes.c_void_p(t.data_ptr()) for t in d + o), len(s1)) == 0
        return [t.cpu().numpy() for t in o]

    return run


def _pairs(rng, n, lo, hi):
    """Same-sign pairs with exponents of either difference in [lo, hi)."""
    m = [rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(lo, hi, n) for _ in range(2)]
    sign = np.where(rng.random(n) < 0.5, -1.0, 1.0)
    return sign * m[0], sign * m[1]


@pytest.mark.parametrize("lo,hi", [(-3, 3), (-60, 60), (-499, 500), (-520, -490), (-545, -500), (490, 512)])
def test_quotient_is_within_an_ulp_of_the_divide(limiter, lo, hi):
    """At most one neighbour away, and away only where the quotient lies within
    2^-12 ulp of a midpoint: one in 2^11 of all, asserted as one in 2^10."""
    s1, s2 = _pairs(np.random.default_rng(abs(hi)), 1 << 20, lo, hi)
    got, ref = limiter(s1, s2)
    with np.errstate(over="ignore"):
        p = s1 * s2
    assert np.isfinite(ref[np.isfinite(p)]).all()
    ok = np.isfinite(ref) & (ref != 0)
    assert np.array_equal(got[~ok], ref[~ok], equal_nan=True)
    away = got[ok] != ref[ok]
    assert (np.abs(got[ok] - ref[ok]) <= np.spacing(np.abs(ref[ok]))).all()
    assert away.mean() <= 2.0 ** -10
    out = p[ok] < 2.0 ** -1000                       # divided: the same
    assert not away[out].any()


def test_error_against_rational_arithmetic(limiter):
    """(1/2 + 2^-12) ulp of the exact quotient of the rounded product and sum."""
    s1, s2 = _pairs(np.random.default_rng(1), 4096, -300, 300)
    s2[:2048] = s1[:2048] * np.random.default_rng(2).uniform(0.5, 2.0, 2048)
    got, _ = limiter(s1, s2)
    for a, b, g in zip(s1, s2, got):
        exact = Fraction(float(a * b)) / Fraction(float(a + b))
        assert abs(Fraction(float(g)) - exact) <= Fraction(float(np.spacing(abs(g)))) * (Fraction(1, 2) + Fraction(1, 4096))


def test_ends_of_the_ranges_and_special_values(limiter):
    """As with the divide, bit for bit: products at and around the smallest normal
    one and the line of the two ways, underflowing and overflowing ones, sums near
    the largest value, zeros, opposite signs, infinities and NaN."""
    e = [0.0, -0.0, 5e-324, 2.0 ** -1074 * 3, 2.0 ** -1022, 2.0 ** -537, 2.0 ** -511, 2.0 ** -500, 1e-160, 1e-154, 1.0, 1.5,
         2.0 ** 511, 2.0 ** 512, 1e160, 2.0 ** 1020, 2.0 ** 1021, 2.0 ** 1022, 1.7e308, np.inf, np.nan]
    e = np.array(e + [-x for x in e])
    a, b = [x.ravel().copy() for x in np.meshgrid(e, e)]
    got, ref = limiter(a, b)
    with np.errstate(all="ignore"):
        p, s = a * b, a + b
    fast = (p >= 2.0 ** -1000) & np.isfinite(p) & (np.abs(s) < 2.0 ** 1021)
    assert np.array_equal(got[~fast], ref[~fast], equal_nan=True)
    assert (np.abs(got[fast] - ref[fast]) <= np.spacing(np.abs(ref[fast]))).all()
    # products of 2^-1000 and its neighbours, and of the smallest normal number
    for k in (-1000, -1022):
        x = 2.0 ** (k // 2)
        a = np.array([x, x, x, np.nextafter(x, 0), np.nextafter(x, 1)])
        b = np.array([x, np.nextafter(x, 0), np.nextafter(x, 1), x, x])
        got, ref = limiter(a, b)
        assert (np.abs(got - ref) <= np.spacing(ref)).all()
