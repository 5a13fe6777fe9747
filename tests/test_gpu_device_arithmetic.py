"""The stream/collide's reciprocal and fixed-point conversion by themselves.

vrcp against CUDA's correctly rounded reciprocal, every significand of every
binade that densities can lie in (2^-60 to 2^60), one and two values wide:
within one unit in the last place.  scat_fixed against the conversion of the
other kernels (f32_to_i64_rn) and against exact integers: nearest, ties to
even, up to 2^63, at and beside the ties between its two 32-bit pieces."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1507_04891_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_lattice.cuh"
using namespace lbm_gb300;
__device__ unsigned long long n_off[4];
__global__ void k_rcp(int e) {
  const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;
  const float x = __uint_as_float((uint32_t)(e + 127) << 23 | m);
  const float y = __uint_as_float((uint32_t)(e + 127) << 23 | (m * 2654435761u & 0x7fffffu));
  V<2> p;
  p.set(0, x);
  p.set(1, y);
  const V<2> w = vrcp<2>(p);
  const float got[3] = {vrcp<1>(V<1>(x)).a, w.get(0), w.get(1)};
  const float want[3] = {__frcp_rn(x), __frcp_rn(x), __frcp_rn(y)};
  for (int k = 0; k < 3; ++k) {
    const int d = abs(__float_as_int(got[k]) - __float_as_int(want[k]));
    if (d) atomicAdd(&n_off[0], 1ull);
    if (d > 1) atomicAdd(&n_off[1], 1ull);
  }
}
__global__ void k_fixed(const float* x, long long* a, long long* b, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  a[i] = (long long)scat_fixed(x[i]);
  b[i] = (long long)f32_to_i64_rn(x[i]);
}
extern "C" int rcp(unsigned long long* off) {
  unsigned long long z[4] = {};
  if (cudaMemcpyToSymbol(n_off, z, sizeof z) != cudaSuccess) return 1;
  for (int e = -60; e <= 60; ++e) k_rcp<<<(1 << 23) / 256, 256>>>(e);
  return (int)cudaMemcpyFromSymbol(off, n_off, 2 * sizeof(off[0]));
}
extern "C" int fixed(const float* x, long long* a, long long* b, int n) {
  float* d = nullptr;
  long long *p = nullptr, *q = nullptr;
  cudaMalloc(&d, n * sizeof(float));
  cudaMalloc(&p, n * sizeof(long long));
  cudaMalloc(&q, n * sizeof(long long));
  cudaMemcpy(d, x, n * sizeof(float), cudaMemcpyHostToDevice);
  k_fixed<<<(n + 255) / 256, 256>>>(d, p, q, n);
  cudaMemcpy(a, p, n * sizeof(long long), cudaMemcpyDeviceToHost);
  const int rc = (int)cudaMemcpy(b, q, n * sizeof(long long), cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(p);
  cudaFree(q);
  return rc;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("arith")
    (d / "a.cu").write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-I", B.CSRC, str(d / "a.cu"), "-o", str(d / "a.so")], check=True,
                   capture_output=True)
    return ctypes.CDLL(os.path.join(str(d), "a.so"))


def test_reciprocal(lib):
    off = (ctypes.c_ulonglong * 2)()
    assert lib.rcp(off) == 0
    assert off[1] == 0  # more than one unit away
    assert off[0] <= 3 * 121  # and away at all: at most one significand of a binade


def test_fixed_point(lib):
    g = np.random.Generator(np.random.PCG64(8))
    x = [np.ldexp(g.uniform(0.5, 1.0, 20000), g.integers(-10, 64, 20000))]
    k = g.integers(0, 1 << 8, 4000).astype(np.float64)
    for half in (0.5, 0.5 - 2.0 ** -12, 0.5 + 2.0 ** -12):
        x.append((k + half) * 2.0 ** 32)  # the rest beside and at half of the upper piece
        x.append(k + half)  # and a tie of the integer
    x = np.concatenate(x + [np.array([0.0, 0.5, 1.5, 2.0 ** 31, 2.0 ** 32 - 256, 2.0 ** 62])])
    x = np.concatenate([x, -x]).astype(np.float32)
    x = x[np.abs(x) < 2.0 ** 63]
    n = len(x)
    a, b = np.zeros(n, np.int64), np.zeros(n, np.int64)
    p = lambda v: v.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    assert lib.fixed(p(x), p(a), p(b), n) == 0
    want = np.array([round(float(v)) for v in x], dtype=np.int64)  # ties to even
    assert np.array_equal(a, want)
    assert np.array_equal(b, want)
