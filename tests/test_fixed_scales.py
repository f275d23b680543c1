"""The kernel shapes of csrc/sph_fixed.cuh near the cutoff, relative to their
own values, in exact integer arithmetic (compiled for the host)."""
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
unsigned f_lead(unsigned long long t) { return lead32(t); }
unsigned long long f_t(unsigned long long r2) { return shape_t(r2); }
unsigned long long f_F(unsigned long long t, unsigned lead) {
  unsigned long long T = scaled_t(t, lead); return mulhi(mulhi(T, T), T); }
unsigned long long f_W8(unsigned long long t, unsigned lead) {
  unsigned long long T = scaled_t(t, lead); return shape_w8(t, mulhi(T, T)); }
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("scales")
    (d / "f.cpp").write_text(SRC)
    so = str(d / "f.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2405_03980_gb300", "csrc"), "-o", so,
                    str(d / "f.cpp")], check=True)
    L = C.CDLL(so)
    u64, u32 = C.c_ulonglong, C.c_uint
    for name, res, args in (("f_lead", u32, [u64]), ("f_t", u64, [u64]), ("f_F", u64, [u64, u32]),
                            ("f_W8", u64, [u64, u32])):
        getattr(L, name).restype = res
        getattr(L, name).argtypes = args
    return L


@pytest.mark.parametrize("t", [0.6, 0.1, 0.03, 0.01, 1e-3, 1e-4, 1e-6, 1e-9])
def test_shapes_keep_their_precision_near_the_cutoff(lib, t):
    """r to one unit of 2^-62 makes t good to 2^-62 / t of itself and its third
    and fourth power three and four times that; the products, truncated at
    2^-64 with T in [1/2, 1), add at most 2^-59 (F above 1/8) and 2^-56.8 (W / 8
    above 1/128, at t near one).  The same holds at the scale of a class whose
    largest t is up to four times as large, relative to that one's shapes."""
    rng = np.random.default_rng(3)
    for _ in range(400):
        r = 1 - Fraction(t) * Fraction(float(rng.uniform(0.6, 1.5)))
        r2 = int(r * r * 2**60)
        exact = 1 - Fraction(math.isqrt(r2 << 128), 2**94)
        got = lib.f_t(r2)
        assert abs(Fraction(got, 2**64) - exact) <= Fraction(5, 2**64)
        off = Fraction(5, 2**64) / exact
        lead = lib.f_lead(got)
        assert 2**63 <= got << lead < 2**64
        F, W = exact**3, exact**4 * (5 - 4 * exact)
        for back in range(0, min(lead, 2) + 1):   # scales of larger neighbours in the class
            f = Fraction(lib.f_F(got, lead - back), 2 ** (64 + 3 * (lead - back)))
            w = Fraction(lib.f_W8(got, lead - back), 2 ** (61 + 4 * (lead - back)))
            assert abs(f / F - 1) <= 3.01 * off + Fraction(2 ** (3 * back), 2**59)
            assert abs(w / W - 1) <= 4.01 * off + Fraction(2 ** (4 * back), 2**56)
