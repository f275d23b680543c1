"""The fixed-point arithmetic of the FP64 form's pair geometry
(csrc/sph_fixed.cuh), compiled for the host and held to exact integer
arithmetic: the bounds below are those stated in the header, in units of the
last place of each result."""
import ctypes as C
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "sph_fixed.cuh"
using namespace sphgb::fx;
extern "C" {
long long f_fixed(double x, double two_h) { return to_fixed(x, make_unit(two_h)); }
unsigned long long f_norm2(long long x, long long y, long long z) { return norm2(split(x), split(y), split(z)); }
long long f_root(unsigned long long r2) { return root(r2); }
unsigned long long f_w8(unsigned long long r2) { unsigned long long t = shape_t(r2); return shape_w8(t, mulhi(t, t)); }
long long f_mul(long long a, long long b) { return mul(split(a), split(b)); }
long long f_cross(long long a, long long b, long long c, long long d) { return mul_sub(split(a), split(b), split(c), split(d)); }
long long f_recip(long long r) { return recip(r); }
double f_sum(const long long* v, const int* s, int n, int e) {
  Acc96 a; for (int k = 0; k < n; ++k) a.add_shifted(v[k], s[k]); return a.value(e); }
long long f_mant(double x, int e) { return mantissa_at(x, e); }
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "f.cpp").write_text(SRC)
    so = str(d / "f.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2405_03980_gb300", "csrc"), "-o", so,
                    str(d / "f.cpp")], check=True)
    L = C.CDLL(so)
    i64, u64, dbl = C.c_longlong, C.c_ulonglong, C.c_double
    for name, res, args in (("f_fixed", i64, [dbl, dbl]), ("f_norm2", u64, [i64] * 3),
                            ("f_root", i64, [u64]), ("f_w8", u64, [u64]),
                            ("f_mul", i64, [i64] * 2), ("f_cross", i64, [i64] * 4),
                            ("f_recip", i64, [i64]), ("f_mant", i64, [dbl, C.c_int]),
                            ("f_sum", dbl, [C.POINTER(i64), C.POINTER(C.c_int), C.c_int, C.c_int])):
        getattr(L, name).restype = res
        getattr(L, name).argtypes = args
    return L


@pytest.mark.parametrize("two_h", [2.6, 1.0, 0.37, 2.0, 5.2e-6, 1e4])
def test_geometry_within_its_units(lib, two_h):
    """Pair vectors exact to 2 units of 2^-62 whatever the distance from the
    origin, r^2 to 3 units of 2^-60 of its own inputs, r to one unit of
    2^-62, W to 1e-17 (shape between 0 and 1)."""
    rng = np.random.default_rng(7)
    for _ in range(1500):
        far = two_h * 2.0 ** int(rng.integers(0, 20))
        xi = rng.uniform(-1, 1, 3) * far
        xj = xi - rng.uniform(-1, 1, 3) * two_h * 0.6
        d = [(lib.f_fixed(a, two_h) - lib.f_fixed(b, two_h) + 2**63) % 2**64 - 2**63
             for a, b in zip(xi, xj)]
        for a, b, q in zip(xi, xj, d):
            assert abs(q - (Fraction(a) - Fraction(b)) / Fraction(two_h) * 2**62) <= 2
        r2 = lib.f_norm2(*d)
        assert abs(r2 - Fraction(sum(q * q for q in d), 2**64)) <= 3
        if not 2**48 <= r2 < 2**60:
            continue
        r = lib.f_root(r2)
        assert abs(r - math.isqrt(r2 << 64)) <= 1
        t = 1 - Fraction(math.isqrt(r2 << 64), 2**62)
        W = t**4 * (5 - 4 * t)
        assert abs(Fraction(lib.f_w8(r2), 2**61) - W) < Fraction(1, 10**17)


def test_products_sums_and_conversions(lib):
    rng = np.random.default_rng(8)
    big = lambda s=0: int(rng.integers(-2**62, 2**62)) >> s  # noqa: E731
    for _ in range(3000):
        a, b, c, d = big(), big(), big(1), big(1)
        assert abs(lib.f_mul(a, b) - Fraction(a * b, 2**64)) <= 2
        assert abs(lib.f_cross(a >> 1, b >> 1, c, d)
                   - Fraction((a >> 1) * (b >> 1) - c * d, 2**64)) <= 3
        rho = int(rng.integers(2**59, 2**62))
        assert abs(lib.f_recip(rho) - Fraction(2**121, rho)) <= 3
        v = [big(int(rng.integers(0, 60))) for _ in range(160)]
        s = [int(rng.integers(0, 25)) for _ in v]
        tot = sum(x << k for x, k in zip(v, s))
        e = int(rng.integers(-200, 100))
        got = lib.f_sum((C.c_longlong * 160)(*v), (C.c_int * 160)(*s), 160, e)
        want = Fraction(tot) * Fraction(2) ** e
        assert abs(Fraction(got) - want) <= abs(want) * Fraction(1, 2**53)
        x = float(rng.normal()) * 2.0 ** int(rng.integers(-40, 40))
        ex = math.frexp(x)[1] + int(rng.integers(0, 70))
        q = Fraction(lib.f_mant(x, ex)) - Fraction(x) * Fraction(2) ** (61 - ex)
        assert abs(q) < 1
    assert lib.f_sum((C.c_longlong * 2)(5, -5), (C.c_int * 2)(3, 3), 2, 0) == 0.0
    assert lib.f_sum((C.c_longlong * 1)(1 << 60), (C.c_int * 1)(0), 1, 2000) == math.inf
    assert lib.f_mant(0.0, 5) == 0 and lib.f_fixed(math.nan, 2.6) == 0
