"""The FP32 register QR alone: a trailing update is rounded once, not once for each of the
panel's sixteen reflectors."""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_07615_gb300", "csrc")

PROGRAM = r"""
#include "qr_reg.cuh"
using namespace tn;
static constexpr int M = 17, N = 17;
__global__ void __launch_bounds__(QRT) run(const float* in, float* Q, float* R, float* Tg) {
  __shared__ __align__(16) float A[M * N];
  __shared__ __align__(16) float V[M * 16];
  __shared__ __align__(16) float part[QR_PART_BYTES / sizeof(float)];
  __shared__ __align__(16) float sm[1024];
  for (int i = threadIdx.x; i < M * N; i += blockDim.x) A[i] = in[i];
  __syncthreads();
  qr_reg(A, M, N, N, Q, N, R, N, V, part, Tg, sm);
}
int main() {
  float h[M * N] = {};
  const float delta = 0x1p-25f;                    // half of half a unit in the last place of 1
  for (int i = 0; i < 16; ++i) { h[i * N + i] = 1.f; h[16 * N + i] = delta; }
  for (int i = 0; i < M; ++i) h[i * N + 16] = 1.5f;
  float *A, *Q, *R, *T;
  if (cudaMalloc(&A, sizeof(h)) || cudaMalloc(&Q, sizeof(h)) || cudaMalloc(&R, sizeof(h)) ||
      cudaMalloc(&T, (16 * N + 256) * sizeof(float)) || cudaMemcpy(A, h, sizeof(h), cudaMemcpyHostToDevice)) return 2;
  run<<<1, QRT>>>(A, Q, R, T);
  if (cudaMemcpy(h, R, sizeof(h), cudaMemcpyDeviceToHost)) return 3;
  printf("%a\n", h[16 * N + 16]);
  return 0;
}
"""


def test_trailing_update_is_rounded_once(tmp_path):
    """Sixteen reflectors that each change the last entry, 1.5, by 1.5 x 2^-25, less than half a unit
    in its last place (2^-24).  R's last entry is that entry, so it may be off by one
    rounding of 1.5 and by the sixteen changes' own relative rounding."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    src, exe = tmp_path / "qr.cu", tmp_path / "qr"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    a = np.zeros((17, 17))
    a[:16, :16] = np.eye(16)
    a[16, :16] = 2.0 ** -25
    a[:, 16] = 1.5
    ref = abs(np.linalg.qr(a)[1][16, 16])
    assert abs(float.fromhex(r.stdout.strip()) - ref) <= 2.0 ** -24 + 16 * 1.5 * 2.0 ** -25 * 1e-6
