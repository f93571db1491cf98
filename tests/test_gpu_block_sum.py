"""The block sum of device_common.cuh takes the pairs of the warps' butterflies:
the bits of the same tree on the host, for every choice of the summing warp."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "device_common.cuh"
__global__ void __launch_bounds__(256) k(const double* v, double* out) {
  __shared__ double sh[8];
  const double x = v[blockIdx.x * 256 + threadIdx.x];
  const double a = erem::block_reduce<0>(x, sh);
  const double b = erem::block_reduce<0>(2.0 * x, sh);   // the buffer again
  if (threadIdx.x == 0) {
    out[2 * blockIdx.x] = a;
    out[2 * blockIdx.x + 1] = b;
  }
}
extern "C" int run(const double* v, double* out, int blocks) {
  double *d, *o;
  if (cudaMalloc(&d, sizeof(double) * 256 * blocks) != cudaSuccess) return 1;
  if (cudaMalloc(&o, sizeof(double) * 2 * blocks) != cudaSuccess) return 1;
  cudaMemcpy(d, v, sizeof(double) * 256 * blocks, cudaMemcpyHostToDevice);
  k<<<blocks, 256>>>(d, o);
  cudaMemcpy(out, o, sizeof(double) * 2 * blocks, cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(o);
  return cudaGetLastError() != cudaSuccess;
}
"""


@pytest.mark.parametrize("span", [0, 40])
def test_block_sum_has_the_bits_of_the_butterflies(tmp_path, span):
    from paper_1209_5553_gb300 import build

    src, so = tmp_path / "m.cu", tmp_path / "m.so"
    src.write_text(SRC)
    subprocess.run([os.path.join(build._cuda_home(), "bin", "nvcc"), *build.ARCH, "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I", build.CSRC, "-o", str(so), str(src)], check=True)
    blocks = 1500
    rng = np.random.default_rng(span)
    v = rng.normal(size=(blocks, 256)) * 2.0 ** rng.integers(-span, span + 1, (blocks, 256))
    v[7, 11], v[8, 200], v[9, 3:5] = np.nan, np.inf, (np.inf, -np.inf)
    out = np.zeros((blocks, 2))
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    assert ctypes.CDLL(str(so)).run(ptr(v), ptr(out), blocks) == 0
    with np.errstate(invalid="ignore"):
        w = v.reshape(blocks, 8, 32)
        for o in (16, 8, 4, 2, 1):
            w = w + w[:, :, np.arange(32) ^ o]
        w = w[:, :, 0]
        for o in (4, 2, 1):
            w = w + w[:, np.arange(8) ^ o]
    assert np.array_equal(out[:, 0], w[:, 0], equal_nan=True)
    assert np.array_equal(out[:, 1], 2.0 * w[:, 0], equal_nan=True)
