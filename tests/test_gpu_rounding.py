"""The branch-free reciprocal and square root of the association against the
IEEE-rounded intrinsics, over every significand of every exponent they are
used at (2^31 and 2^30 values, a fraction of a second on the GPU)."""
import importlib
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "kf_icp.cuh"
#include <cstdio>
using namespace kf;
__global__ void check(int exponent, unsigned long long* bad) {
  const unsigned m = blockIdx.x * 256u + threadIdx.x;
  const float v = __int_as_float((exponent << 23) | (int)m);
  if (exponent <= 252 && __float_as_int(rcp_rn_mid(v)) != __float_as_int(__frcp_rn(v))) atomicAdd(bad, 1ull);
  if (exponent >= 27 && __float_as_int(sqrt_rn_mid(v)) != __float_as_int(__fsqrt_rn(v))) atomicAdd(bad + 1, 1ull);
}
int main() {
  unsigned long long *d, h[2];
  if (cudaMalloc(&d, 16) != cudaSuccess || cudaMemset(d, 0, 16) != cudaSuccess) return 2;
  for (int e = 1; e <= 254; ++e) check<<<(1 << 23) / 256, 256>>>(e, d);
  if (cudaMemcpy(h, d, 16, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  printf("%llu %llu\n", h[0], h[1]);
  return 0;
}
"""


def test_every_significand_rounds_as_the_intrinsics(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B = importlib.import_module("paper_1802_03980_gb300.build")
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(SRC)
    subprocess.run([B.nvcc()] + B.flags() + [str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["0", "0"]
