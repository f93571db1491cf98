"""The device helpers that replace FP64 divisions and roots (device_common.cuh)
against the compiler's own, compiled here from the library's header."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "device_common.cuh"
__global__ void k(const double* a, const double* b, double* q, double* r, double* s, double* t, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    q[i] = erem::div_newton(a[i], b[i]);
    r[i] = a[i] / b[i];
    s[i] = erem::sqrt_newton(a[i]);
    t[i] = sqrt(a[i]);
  }
}
extern "C" int run(const double* a, const double* b, double* q, double* r, double* s, double* t, int n) {
  double* d[6];
  const double* in[2] = {a, b};
  double* out[4] = {q, r, s, t};
  for (int j = 0; j < 6; ++j)
    if (cudaMalloc(&d[j], sizeof(double) * n) != cudaSuccess) return 1;
  for (int j = 0; j < 2; ++j) cudaMemcpy(d[j], in[j], sizeof(double) * n, cudaMemcpyHostToDevice);
  k<<<1024, 256>>>(d[0], d[1], d[2], d[3], d[4], d[5], n);
  for (int j = 0; j < 4; ++j) cudaMemcpy(out[j], d[2 + j], sizeof(double) * n, cudaMemcpyDeviceToHost);
  for (int j = 0; j < 6; ++j) cudaFree(d[j]);
  return cudaGetLastError() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1209_5553_gb300 import build

    nvcc = os.path.join(build._cuda_home(), "bin", "nvcc")
    assert os.path.exists(nvcc) or shutil.which("nvcc")
    d = tmp_path_factory.mktemp("math")
    src, so = d / "m.cu", d / "m.so"
    src.write_text(SRC)
    subprocess.run([nvcc, *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC,
                    "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def run(lib, a, b):
    a, b = np.ascontiguousarray(a), np.ascontiguousarray(b)
    out = [np.zeros(a.size) for _ in range(4)]
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    assert lib.run(ptr(a), ptr(b), *[ptr(o) for o in out], a.size) == 0
    return out


@pytest.mark.parametrize("span", [0.0, 2.0, 60.0, 300.0])
def test_div_and_sqrt_against_the_compilers(lib, span):
    rng = np.random.default_rng(int(span) + 1)
    n = 4_000_000
    a = rng.uniform(1, 2, n) * 2.0 ** np.round(rng.uniform(-span, span, n))
    b = rng.uniform(1, 2, n) * 2.0 ** np.round(rng.uniform(-span, span, n)) * rng.choice([-1.0, 1.0], n)
    # significands next to powers of two and to each other
    k = n // 8
    b[:k] = np.nextafter(np.abs(b[:k]) // 1 + 1.0, rng.choice([0.0, 1e300], k))
    a[k:2 * k] = b[k:2 * k] * (1 + rng.integers(-3, 4, k) * 2.0**-52)
    q, r, s, t = run(lib, a, b)
    d = np.abs(q - r) / np.spacing(np.abs(r))
    assert d.max() <= 1.0 and (d > 0).sum() <= 2       # about 1e-10 of the pairs
    pos = a > 0
    assert (np.abs(s[pos] - t[pos]) <= 2 * np.spacing(t[pos])).all()


def test_div_and_sqrt_special_values(lib):
    v = np.array([0.0, -0.0, 1.0, -1.0, 3.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, -1e-310, 1e308, 2.2e-308,
                  1e-160, 1e160, 2.0**500, 2.0**-500, 2.0**501, 2.0**-501])
    a, b = (x.ravel() for x in np.meshgrid(v, v))
    q, r, s, t = run(lib, a, b)
    assert np.array_equal(q, r, equal_nan=True)
    assert np.allclose(s, t, rtol=4.5e-16, atol=0, equal_nan=True)
