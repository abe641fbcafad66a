"""The block reduction of csrc/common.cuh over every block size it takes: 32 to 1024 threads."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1005_0542_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "common.cuh"
template <int NV>
__global__ void sum_kernel(const double *x, double *out) {
  double v[NV];
  for (int i = 0; i < NV; ++i) v[i] = x[i * blockDim.x + threadIdx.x];
  lag::block_sum<NV>(v);
  if (threadIdx.x == 0)
    for (int i = 0; i < NV; ++i) out[i] = v[i];
}
extern "C" int block_sums(const double *x, int threads, int nv, double *out) {
  double *d = nullptr;
  if (cudaMalloc(&d, (nv * threads + nv) * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(d, x, nv * threads * sizeof(double), cudaMemcpyHostToDevice);
  if (nv == 1) sum_kernel<1><<<1, threads>>>(d, d + threads);
  else sum_kernel<2><<<1, threads>>>(d, d + 2 * threads);
  const int rc = cudaMemcpy(out, d + nv * threads, nv * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return rc;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("block_sum")
    src, so = d / "block_sum.cu", d / "block_sum.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", str(so), str(src)],
                   check=True, cwd=os.path.dirname(str(src)))
    return C.CDLL(str(so))


# whole numbers: every order of additions gives the same sum
@pytest.mark.parametrize("nv", [1, 2])
@pytest.mark.parametrize("threads", [32, 64, 96, 192, 256, 288, 512, 544, 992, 1024])
def test_block_sum(lib, threads, nv):
    x = np.random.default_rng(threads).integers(-2 ** 40, 2 ** 40, (nv, threads)).astype(np.float64)
    out = np.zeros(nv)
    assert lib.block_sums(x.ctypes.data_as(C.c_void_p), threads, nv, out.ctypes.data_as(C.c_void_p)) == 0
    assert np.array_equal(out, x.sum(axis=1))
