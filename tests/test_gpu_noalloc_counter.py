"""Each call of kf_reduce_noalloc starts its arrivals from zero, whatever an
earlier one left in the shared array: direct calls and a replayed capture give
the first call's sums after the array's header was overwritten.
"""
import importlib
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "kf_icp.cu"
#include <cmath>
#include <cstdio>
#include <vector>
using namespace kf;
#define CK(x) do { if ((x) != cudaSuccess) { printf("line %d\n", __LINE__); return 2; } } while (0)
int main() {
  const int w = 320, h = 240, n = w * h;
  std::vector<float> v(3 * n), nn(3 * n);
  for (int i = 0; i < n; ++i) {
    const float z = 2.f + 0.001f * (i % 7);
    v[3 * i] = (i % w - 160.f) / 250.f * z;
    v[3 * i + 1] = (i / w - 120.f) / 250.f * z;
    v[3 * i + 2] = z;
    nn[3 * i] = nn[3 * i + 1] = 0.1f;
    nn[3 * i + 2] = -std::sqrt(0.98f);
  }
  float *dv, *dn;
  double* out;
  CK(cudaMalloc(&dv, 12 * n));
  CK(cudaMalloc(&dn, 12 * n));
  CK(cudaMalloc(&out, 29 * sizeof(double)));
  CK(cudaMemcpy(dv, v.data(), 12 * n, cudaMemcpyHostToDevice));
  CK(cudaMemcpy(dn, nn.data(), 12 * n, cudaMemcpyHostToDevice));
  cudaStream_t s;
  CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  kf_intrinsics K = {w, h, 250.0, 250.0, 160.0, 120.0};
  double T[16] = {1, 0, 0, 0.003, 0, 1, 0, 0.001, 0, 0, 1, -0.002, 0, 0, 0, 1}, M[16] = {1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1};
  auto call = [&] { return kf_reduce_noalloc(dv, w, h, dv, dn, &K, T, M, 0.16, 512, 0, 400, out, s); };
  auto clear = [&] { return cudaMemsetAsync(out, 0xff, 29 * sizeof(double), s); };
  double want[29], got[29];
  auto same = [&] {
    if (cudaMemcpyAsync(got, out, sizeof(got), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) return false;
    return memcmp(got, want, sizeof(got)) == 0;
  };
  // the header's first words: arrivals that calls which overlapped, early ones
  // here, may leave
  void* head;
  CK(cudaGetSymbolAddress(&head, g_noalloc_scratch));
  auto plant = [&] {
    std::vector<unsigned> left(64, 3u);
    for (int i = 0; i < 64; i += 2) left[i] = 1000u;
    return cudaMemcpyAsync(head, left.data(), 256, cudaMemcpyHostToDevice, s);
  };
  for (int i = 0; i < 8; ++i)
    if (call() != KF_OK) return 3;
  CK(cudaMemcpyAsync(want, out, sizeof(want), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  if (!(want[27] > 0.5 * n)) return 4;
  cudaGraph_t g;
  cudaGraphExec_t x;
  CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeGlobal));
  if (call() != KF_OK) return 3;
  CK(cudaStreamEndCapture(s, &g));
  CK(cudaGraphInstantiate(&x, g, 0));
  int bad = 0;
  for (int i = 0; i < 6; ++i) {
    CK(clear());
    if (i & 1) CK(plant());
    if (i < 4) CK(cudaGraphLaunch(x, s));
    else if (call() != KF_OK) return 3;
    if (!same()) ++bad;
  }
  printf("%d differ\n", bad);
  return 0;
}
"""


def test_every_call_starts_from_zero(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B = importlib.import_module("paper_1802_03980_gb300.build")
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(SRC)
    subprocess.run([B.nvcc()] + B.flags() + [str(src), os.path.join(B.CSRC, "kf_team.cu"), "-o", str(exe)],
                   check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert (r.returncode, r.stdout.split()) == (0, ["0", "differ"]), (r.returncode, r.stdout)
