"""The device branches of csrc/sph_fixed.cuh (approximate reciprocals, carry
chains, high products, funnel shifts) in a kernel of their own: the integer
functions equal the host branches, which test_fixed_point.py holds to exact
arithmetic, bit for bit; the two that start from a hardware estimate keep that
test's bounds."""
import ctypes as C
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2405_03980_gb300 import build as Bld
from test_gpu_fp64 import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu

IN, OUT = 10, 11
SRC = r'''
#include <cuda_runtime.h>
#include "sph_fixed.cuh"
using namespace sphgb::fx;
SPH_FX void all(const i64* v, i64* o) {
  const Unit U = {(u64)v[6], (u64)v[7], (int)v[8]};
  Half a[3], b[3];
  for (int k = 0; k < 3; ++k) {
    a[k] = split(v[2 + k] >> 1);
    b[k] = split(v[3 + k] >> 1);
  }
  o[0] = root((u64)v[0]);
  o[1] = recip(v[1]);
  o[2] = mul(split(v[2]), split(v[3]));
  o[3] = mul_sub(a[0], b[0], a[1], b[1]);
  o[4] = dot3(a, b);
  o[5] = (i64)norm2(a[0], a[1], a[2]);
  o[6] = to_fixed(of_bits((u64)v[9]), U);
  o[7] = mantissa_at(of_bits((u64)v[9]), exponent_of(of_bits((u64)v[9])) + (int)(v[2] & 63));
  Sum96 s;
  Acc96 c;
  for (int k = 0; k < 40; ++k) {
    s.add((u64)v[2 + k % 4] * (u64)(2 * k + 1));
    c.add_shifted(v[2 + k % 4] >> (k + 2), (int)(v[3] >> k & 31) % 25);
    c.add(v[5 - k % 4]);
  }
  o[8] = (i64)bits_of(s.shape_sum());
  o[9] = (i64)bits_of(c.value((int)(v[4] & 255) - 128));
  o[10] = (i64)(lead32((u64)v[0]) | (lead32((u64)v[5] >> (v[2] & 63)) << 8));
}
__global__ void k_all(int n, const i64* v, i64* o) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) all(v + (long long)i * IN, o + (long long)i * OUT);
}
extern "C" int run(int n, const i64* v, i64* host, i64* device) {
  i64 *dv = nullptr, *dout = nullptr;
  const size_t bi = sizeof(i64) * IN * (size_t)n, bo = sizeof(i64) * OUT * (size_t)n;
  for (int i = 0; i < n; ++i) all(v + (long long)i * IN, host + (long long)i * OUT);
  int e = cudaMalloc(&dv, bi) || cudaMalloc(&dout, bo) ||
          cudaMemcpy(dv, v, bi, cudaMemcpyHostToDevice);
  if (!e) {
    k_all<<<(n + 127) / 128, 128>>>(n, dv, dout);
    e = cudaGetLastError() || cudaMemcpy(device, dout, bo, cudaMemcpyDeviceToHost);
  }
  cudaFree(dv);
  cudaFree(dout);
  return e;
}
'''


def test_device_branches(tmp_path):
    src, so = tmp_path / "f.cu", str(tmp_path / "f.so")
    src.write_text(f"#define IN {IN}\n#define OUT {OUT}\n" + SRC)
    subprocess.run([Bld.nvcc()] + Bld.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler",
                                             "-fPIC", "-I", Bld.CSRC, "-o", so, str(src)],
                   check=True)
    rng = np.random.default_rng(4)
    n = 20000
    v = np.zeros((n, IN), dtype=np.int64)
    v[:, 0] = np.exp2(rng.uniform(48, 60, n)).astype(np.int64)
    v[:, 1] = rng.integers(2**59, 2**62, n)
    v[:, 2:6] = rng.integers(-2**62, 2**62, (n, 4)) >> rng.integers(0, 50, (n, 4))
    for k, two_h in enumerate((2.6, 1.0, 5.2e-6, 1e4)):  # r1, r0, eh of fx::make_unit
        m, e = math.frexp(two_h)
        q = (2**180 - 1) // int(m * 2**53)
        v[k::4, 6:9] = np.array([q >> 64, q & (2**64 - 1), (e - 53) % 2**64],
                                dtype=np.uint64).view(np.int64)
        v[k::4, 9] = (rng.normal(size=v[k::4].shape[0]) * two_h
                      * 10.0 ** rng.uniform(-20, 6, v[k::4].shape[0])).view(np.int64)
    v[:6, 0] = [2**48, 2**48 + 1, 2**54 - 1, 2**54, 2**60 - 1, 2**59]
    v[:3, 1] = [2**59, 2**62, 2**62 - 1]
    v[6:12, 9] = np.array([0.0, -0.0, 5e-324, np.inf, -np.inf, np.nan]).view(np.int64)
    host, dev = np.zeros((n, OUT), dtype=np.int64), np.zeros((n, OUT), dtype=np.int64)
    lib = C.CDLL(so)
    p = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    assert lib.run(n, p(v), p(host), p(dev)) == 0
    assert np.array_equal(dev[:, 2:], host[:, 2:])
    for i in range(n):
        r2, rho = int(v[i, 0]), int(v[i, 1])
        assert abs(int(dev[i, 0]) - math.isqrt(r2 << 64)) <= 1
        assert abs(int(dev[i, 1]) - Fraction(2**121, rho)) <= 3
