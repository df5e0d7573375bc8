"""Device functions of the library one by one (device_probe.cu), against exact arithmetic."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2408_00598_gb300 import build
    out = str(tmp_path_factory.mktemp("probe") / "libprobe.so")
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-Xcompiler", "-fvisibility=default", "-I" + build.CSRC,
                    "-shared", "-o", out, os.path.join(HERE, "device_probe.cu")], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("S", [33, 64])
@pytest.mark.parametrize("span", [1.0, 700.0])
@pytest.mark.parametrize("size", [1e-12, 1e-6, 1.0])
def test_fp64_reduced_cost_error_is_relative_to_the_element(probe, S, span, size):
    """g = h (x_r - x_c)^2 - alpha - beta with real-valued positions: the rounding of the difference (2 u c), of
    c - alpha and of g, each once; nothing relative to the largest cost of the grid.  alpha and beta of `size`
    largest costs, so that c is small against the largest cost wherever g < 0."""
    rng = np.random.default_rng(S)
    X = np.sort(rng.random(S)) * span
    h = 2.0 ** -int(np.ceil(np.log2((X[-1] - X[0]) ** 2)))
    ab = size * (0.5 + 0.5 * rng.random(2 * S))
    out = np.zeros((S, S))
    assert probe.probe_sweep64(S, ctypes.c_double(h), _ptr(X), _ptr(ab), _ptr(out)) == 0
    u, hf = Fraction(1, 2 ** 53), Fraction(h)
    seen = 0
    for r in range(S):
        for c in range(S):
            cost = hf * (Fraction(X[r]) - Fraction(X[c])) ** 2
            g = cost - Fraction(ab[r]) - Fraction(ab[S + c])
            if g >= 0:
                assert out[r, c] == 0.0
                continue
            seen += 1
            bound = u * (2 * cost + abs(cost - Fraction(ab[r])) + abs(g)) * (1 + 8 * u)
            assert abs(Fraction(out[r, c]) + g) <= bound, (r, c)
    assert seen >= S


def _two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def _pair_add(ah, al, b):
    s, e = _two_sum(ah, b)
    e = e + al
    h = s + e
    return h, e - (h - s)


@pytest.mark.parametrize("terms", [1, 5, 64])
@pytest.mark.parametrize("square", [True, False])
def test_sums_of_products_are_sums_of_renormalised_pairs(probe, terms, square):
    """df_dot against the pair sum restated in numpy FP32 (each exact product added as a pair), bit for bit."""
    f4 = np.float32
    rng = np.random.default_rng(terms)
    sums = 4000
    x = (rng.standard_normal((sums, terms)) * 10.0 ** rng.uniform(-3, 3, (sums, terms))).astype(f4)
    y = x if square else rng.standard_normal((sums, terms)).astype(f4)
    hi, lo = np.zeros(sums, f4), np.zeros(sums, f4)
    assert probe.probe_dot(_ptr(x), _ptr(np.ascontiguousarray(y)), terms, sums, _ptr(hi), _ptr(lo)) == 0
    h = np.zeros(sums, f4)
    l = np.zeros(sums, f4)
    for q in range(terms):
        exact = x[:, q].astype(np.float64) * y[:, q]              # exact: 24 + 24 bits
        p = exact.astype(f4)
        pe = (exact - p).astype(f4)
        h, l = _pair_add(*_pair_add(h, l, p), pe)
    np.testing.assert_array_equal(hi, h)
    np.testing.assert_array_equal(lo, l)
