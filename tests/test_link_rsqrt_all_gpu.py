"""The sample rollouts' reciprocal square root (link_rsqrt<true>) against
rsqrtf over every value a squared link length can take: all non-negative FP32
numbers, infinity and the NaNs.  The same bits everywhere but for a subnormal
argument, where it gives infinity -- what the exact second pass relies on."""
import ctypes
import subprocess

import pytest

from paper_2512_04579_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "common.cuh"
using namespace gnm;
// counts[0]: differing values, [1]: subnormal arguments without infinity, [2]: arguments seen
__global__ void scan(unsigned int hi, unsigned long long* counts) {
  unsigned long long c0 = 0, c1 = 0, c2 = 0;
  const unsigned long long n = (unsigned long long)hi + 1, step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n; i += step) {
    const float q = __uint_as_float((unsigned int)i);
    const float a = link_rsqrt<true>(q), b = link_rsqrt<false>(q);
    ++c2;
    if (i > 0 && i < 0x00800000u) {
      if (__float_as_uint(a) != 0x7F800000u || !isfinite(b)) ++c1;
    } else if (isnan(a) != isnan(b) || (!isnan(a) && __float_as_uint(a) != __float_as_uint(b))) {
      ++c0;
    }
  }
  atomicAdd(counts, c0);
  atomicAdd(counts + 1, c1);
  atomicAdd(counts + 2, c2);
}
extern "C" int run(unsigned int hi, unsigned long long* out) {
  unsigned long long* d;
  if (cudaMalloc(&d, 24) != cudaSuccess || cudaMemset(d, 0, 24) != cudaSuccess) return 1;
  scan<<<1216, 256>>>(hi, d);
  const int rc = cudaMemcpy(out, d, 24, cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(d);
  return rc;
}
"""


def test_every_squared_length(tmp_path):
    src, out = tmp_path / "scan.cu", tmp_path / "scan.so"
    src.write_text(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", str(src), "-o", str(out)], check=True)
    counts = (ctypes.c_ulonglong * 3)()
    assert ctypes.CDLL(str(out)).run(0x7FFFFFFF, counts) == 0
    assert counts[2] == 1 << 31
    assert counts[0] == 0 and counts[1] == 0
