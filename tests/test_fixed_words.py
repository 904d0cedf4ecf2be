"""The fixed-point words of fixed.cuh, compiled for the host with CUDA's bit casts spelled out: encoding and
decoding, exact dot products, and the largest number of terms.

Bars.  A word is the value to 2^(E - 1080) (half its last place): encode and decode are off by that plus the
rounding to double.  A dot product of words is exact before its one rounding, apart from what the low sum
loses below 2^29 of the product unit."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1512_00616_gb300", "csrc")
SRC = r"""
#include <algorithm>
#include <cmath>
#include <cstring>
using std::fma; using std::max; using std::min;
#define __device__
#define __forceinline__ inline
#define __align__(n) alignas(n)
template <class B, class A> inline B bits(A a) { B b; std::memcpy(&b, &a, sizeof b); return b; }
inline long long __double_as_longlong(double v) { return bits<long long>(v); }
inline double __longlong_as_double(long long v) { return bits<double>(v); }
inline int __double2hiint(double v) { return (int)(bits<long long>(v) >> 32); }
inline double __hiloint2double(int hi, int lo) { return bits<double>(((long long)hi << 32) | (unsigned)lo); }
inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
#include "fixed.cuh"
using namespace pp;
extern "C" {
int group(int n, const double* x) { int e = 0; for (int i = 0; i < n; ++i) e = max(e, fix_exponent(x[i])); return e; }
void encode(int n, const double* x, int e, int* w) {
  for (int i = 0; i < n; ++i) { Fix q = fix_encode(x[i], e); w[2 * i] = q.hi; w[2 * i + 1] = q.lo; }
}
double decode(const int* w, int e) { return fix_decode(Fix{w[0], w[1]}, e); }
double dot(int n, const int* a, const int* b, int ea, int eb, double s) {
  FixDot acc; acc.clear();
  for (int i = 0; i < n; ++i) acc.add(Fix{a[2 * i], a[2 * i + 1]}, Fix{b[2 * i], b[2 * i + 1]});
  return acc.result(ea + eb, ea == 0x7ff || eb == 0x7ff, s);
}
double dot_small(int n, const int* a, const int* b, int ea, int eb, double s) {
  FixDot acc; acc.clear();
  for (int i = 0; i < n; ++i) acc.add(Fix{a[2 * i], a[2 * i + 1]}, Fix{b[2 * i], b[2 * i + 1]});
  return acc.result<true>(ea + eb, ea == 0x7ff || eb == 0x7ff, s);
}
}
"""
LIMIT = 63   # most terms of a sum (60 are used: block rows, basis vectors, the parts of fix_dot)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "fixed.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-ffp-contract=off", "-I" + CSRC, str(d / "fixed.cpp"),
                    "-o", str(d / "fixed.so")], check=True)
    L = ctypes.CDLL(str(d / "fixed.so"))
    for f in (L.decode, L.dot, L.dot_small):
        f.restype = ctypes.c_double
    return L


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _encode(lib, x, e=None):
    x = np.ascontiguousarray(x, dtype=np.float64)
    e = lib.group(len(x), _p(x)) if e is None else e
    w = np.zeros(2 * len(x), dtype=np.int32)
    lib.encode(len(x), _p(x), e, _p(w))
    return w, e


def _exact(w, e):
    """The words as rationals."""
    return [((int(h) << 29) + int(l)) * Fraction(2) ** (int(e) - 1079) for h, l in zip(w[::2], w[1::2])]


def _ulp(x):
    return Fraction(float(np.spacing(abs(float(x))))) if x else Fraction(2) ** -1074


@pytest.mark.parametrize("scale", [-900, -500, -60, 0, 60, 900])
@pytest.mark.parametrize("spread", [0, 3, 4, 5, 30, 53, 57, 58, 80])
def test_words_hold_58_bits_of_the_group(lib, scale, spread):
    rng = np.random.default_rng(spread)
    x = np.ldexp(rng.uniform(-1.0, 1.0, 64), scale - rng.integers(0, spread + 1, 64))
    x[0] = np.ldexp(1.9, scale)
    x[1] = -np.ldexp(2.0 - 2.0 ** -52, scale)
    w, e = _encode(lib, x)
    assert np.all(np.abs(w[::2]) <= 2 ** 28) and np.all(w[1::2] >= -2 ** 28) and np.all(w[1::2] < 2 ** 28)
    half = Fraction(2) ** (e - 1080)
    for i, q in enumerate(_exact(w, e)):
        if abs(x[i]) < 2.0 ** -1022:
            assert q == 0
            continue
        assert abs(q - Fraction(x[i])) <= half
        if abs(x[i]) >= np.ldexp(1.0, scale - 4):
            assert q == Fraction(x[i])       # within a factor 16 of the largest: all 53 bits
        assert abs(Fraction(lib.decode(_p(w[2 * i:2 * i + 2]), e)) - q) <= _ulp(q) / 2


def test_zeros_and_subnormals_count_as_zero(lib):
    w, e = _encode(lib, [0.0, -0.0, 5e-324, -2.0 ** -1023])
    assert e == 0 and not w.any() and lib.decode(_p(w), e) == 0.0
    w, e = _encode(lib, [1.0, 0.0, 5e-324])
    assert _exact(w, e) == [1, 0, 0]


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_infinities_and_nan_make_results_nan(lib, bad):
    w, e = _encode(lib, [1.0, bad, 0.0])
    one, e1 = _encode(lib, [1.0, 2.0, 3.0])
    zero, e0 = _encode(lib, [0.0, 0.0, 0.0])
    assert e == 0x7ff and np.isnan(lib.decode(_p(w), e))
    for other, eo in ((one, e1), (zero, e0), (w, e)):
        for a, b, ea, eb in ((w, other, e, eo), (other, w, eo, e)):
            assert np.isnan(lib.dot(3, _p(a), _p(b), ea, eb, ctypes.c_double(1.0)))


@pytest.mark.parametrize("n", [1, 2, 12, 15, 40, LIMIT])
@pytest.mark.parametrize("spread", [0, 8, 40])
def test_dots_are_exact_before_their_rounding(lib, n, spread):
    rng = np.random.default_rng(n + spread)
    for scale in (-400, 0, 400, -1000):    # the last: sums below the words' unit in the normal range
        f = lib.dot_small if scale == -1000 else lib.dot
        a = np.ldexp(rng.uniform(-1.0, 1.0, n), scale - rng.integers(0, spread + 1, n))
        b = np.ldexp(rng.uniform(-1.0, 1.0, n), rng.integers(0, spread + 1, n))
        (wa, ea), (wb, eb) = _encode(lib, a), _encode(lib, b)
        for s in (0.0, float(np.ldexp(rng.uniform(), scale))):
            ref = Fraction(s) + sum((x * y for x, y in zip(_exact(wa, ea), _exact(wb, eb))), Fraction(0))
            got = Fraction(f(n, _p(wa), _p(wb), ea, eb, ctypes.c_double(s)))
            # the conversion of the sum and the addition of s round once each
            assert abs(got - ref) <= _ulp(ref - Fraction(s)) / 2 + _ulp(ref) / 2 + Fraction(2) ** (ea + eb - 2158 + 29)


@pytest.mark.parametrize("sign", [1, -1])
def test_the_largest_sums_do_not_overflow(lib, sign):
    """Every term of the largest size and of one sign; hi hi, hi lo + lo hi and lo lo at their largest alike."""
    for hi, lo in ((2 ** 28, -2 ** 28), (2 ** 28, 0), (2 ** 28 - 1, 2 ** 28 - 1), (2 ** 28 - 1, -2 ** 28)):
        w = np.array([hi, lo] * LIMIT, dtype=np.int32)
        u = np.array([sign * hi, max(sign * lo, -2 ** 28)] * LIMIT, dtype=np.int32)
        e = 1079
        ref = sum(x * y for x, y in zip(_exact(w, e), _exact(u, e)))
        assert abs(Fraction(lib.dot(LIMIT, _p(w), _p(u), e, e, ctypes.c_double(0.0))) - ref) <= _ulp(ref)
