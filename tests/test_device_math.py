"""Device arithmetic of gf_complex.cuh against FP64 and exact rationals: a small kernel per function, compiled here."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1111_2157_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "gf_complex.cuh"
namespace cx = gf::cx;
// one thread per row of n values: their sum as a pair, both components of the packed form
__global__ void k_pair_sum(const float* v, int rows, int n, double* out) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= rows) return;
  float2 h = make_float2(0.f, 0.f), l = h;
  for (int i = 0; i < n; ++i) cx::pair2_add(h, l, make_float2(v[r * n + i], -v[r * n + n - 1 - i]));
  out[2 * r] = cx::widen(h.x) + cx::widen(l.x);
  out[2 * r + 1] = cx::widen(h.y) + cx::widen(l.y);
}
__global__ void k_rcp(const double* x, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = cx::rcp_newton(x[i]);
}
__global__ void k_widen(const float* x, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = cx::widen(x[i]);
}
template <class F>
static int run(const void* in, size_t n_in, void* out, size_t n_out, F launch) {
  void *a = nullptr, *b = nullptr;
  if (cudaMalloc(&a, n_in) || cudaMalloc(&b, n_out)) return 1;
  int e = cudaMemcpy(a, in, n_in, cudaMemcpyHostToDevice);
  launch(a, b);
  e |= cudaGetLastError();
  e |= cudaMemcpy(out, b, n_out, cudaMemcpyDeviceToHost);
  cudaFree(a);
  cudaFree(b);
  return e;
}
extern "C" int pair_sum(const float* v, int rows, int n, double* out) {
  return run(v, sizeof(float) * rows * n, out, 16 * rows, [&](void* a, void* b) {
    k_pair_sum<<<(rows + 127) / 128, 128>>>((const float*)a, rows, n, (double*)b);
  });
}
extern "C" int rcp(const double* x, int n, double* out) {
  return run(x, 8 * n, out, 8 * n, [&](void* a, void* b) {
    k_rcp<<<(n + 127) / 128, 128>>>((const double*)a, n, (double*)b);
  });
}
extern "C" int widen(const float* x, int n, double* out) {
  return run(x, 4 * n, out, 8 * n, [&](void* a, void* b) {
    k_widen<<<(n + 127) / 128, 128>>>((const float*)a, n, (double*)b);
  });
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("device_math")
    (d / "t.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", str(d / "t.cu"), "-o", str(d / "t.so")],
                   check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("n", [1, 2, 16, 300])
def test_pair_sums_hold_48_bits(lib, n):
    """Each two_sum is exact and its error is summed in FP32: n 2^-24 of the errors, which are 2^-24 of the partial
    sums, n 2^-48 of the sum of the moduli in all."""
    rng = np.random.default_rng(n)
    rows = 512
    v = (rng.standard_normal((rows, n)) * np.exp(rng.uniform(-12, 3, (rows, n)))).astype(np.float32)
    v[0] = np.float32(1.0 / 3.0)
    out = np.zeros((rows, 2))
    assert lib.pair_sum(_ptr(v), rows, n, _ptr(out)) == 0
    d = v.astype(np.float64)
    for c, ref in enumerate((d.sum(1), -d.sum(1))):
        assert np.all(np.abs(out[:, c] - ref) <= n * 2.0**-48 * np.abs(d).sum(1))


def test_reciprocal_within_one_unit_in_the_last_place(lib):
    """Against numpy's quotient, which is rounded correctly, over every binade whose reciprocal is normal; 0 and
    infinity where the seed is, as the quotient for zero and infinity."""
    rng = np.random.default_rng(0)
    e = np.arange(-1021, 1022)
    x = np.ldexp(1.0 + rng.random((200, e.size)), e).reshape(-1)
    x = np.concatenate([x, -x, np.ldexp(1.0, e), np.ldexp(np.nextafter(2.0, 0.0), e[:-1])])
    x = x[np.abs(x) < 2.0**1021]
    out = np.zeros_like(x)
    assert lib.rcp(_ptr(x), x.size, _ptr(out)) == 0
    q = 1.0 / x
    assert np.all(np.abs(out - q) <= np.spacing(np.abs(q)))
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e308, -1.7e308, 5e-324, -2e-308])
    out = np.zeros_like(x)
    assert lib.rcp(_ptr(x), x.size, _ptr(out)) == 0
    assert np.array_equal(out, [np.inf, -np.inf, 0.0, -0.0, np.nan, 0.0, -0.0, np.inf, -np.inf], equal_nan=True)


def test_widen_is_exact(lib):
    rng = np.random.default_rng(1)
    x = rng.integers(0, 2**32, 200000, dtype=np.uint64).astype(np.uint32).view(np.float32)
    x = np.concatenate([x, np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1.2e-38, 3.4e38], np.float32)])
    out = np.zeros(x.size)
    assert lib.widen(_ptr(x), x.size, _ptr(out)) == 0
    with np.errstate(invalid="ignore"):  # (signalling NaN)
        ref = np.where(np.abs(x) < np.float32(2.0**-126), np.copysign(0.0, x), x.astype(np.float64))  # (denormals: 0)
    assert np.array_equal(out, ref, equal_nan=True)
