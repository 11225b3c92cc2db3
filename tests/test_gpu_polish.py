"""The orthogonalisation of refined columns alone, on one CTA: it keeps the product W V^T, and leaves
columns that are too close for it, saying so."""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_07615_gb300", "csrc")
N, LEN = 24, 40

PROGRAM = r"""
#include "refine64.cuh"
using namespace tn;
static constexpr int N = %d, LEN = %d, SMEM = 64 * 1024;
__global__ void __launch_bounds__(512) run(double* W, double* V, double* V2, float* J, double* nrm, float* stat, int* status,
                                           float tol2, int* out) {
  __shared__ ClusterShared s_cl;
  ClusterCtx cc;
  cl_init(cc, &s_cl, status, 1000000000LL);
  RefineMem<double> m{};
  m.V = V; m.V2 = V2; m.W = W; m.J = J; m.nrm = nrm; m.stat = stat;
  m.ldv = N; m.ldw = LEN; m.ldj = N;
  const int r = rf_polish<double>(cc, m, N, LEN, 1e-27f, tol2, 0, SMEM);
  __syncthreads();
  if (m.V != V)
    for (int i = threadIdx.x; i < N * N; i += blockDim.x) V[i] = m.V[i];
  if (threadIdx.x == 0) *out = r;
}
int main(int argc, char** argv) {
  static double w[N * LEN], v[N * N], q[N];
  FILE* f = fopen(argv[1], "rb");
  if (!f || fread(w, sizeof(w), 1, f) != 1 || fread(v, sizeof(v), 1, f) != 1) return 2;
  fclose(f);
  for (int j = 0; j < N; ++j) { q[j] = 0; for (int i = 0; i < LEN; ++i) q[j] += w[j * LEN + i] * w[j * LEN + i]; }
  double *W, *V, *V2, *nrm;
  float *J, *stat;
  int *st, *out, r = -1;
  if (cudaMalloc(&W, sizeof(w)) || cudaMalloc(&V, sizeof(v)) || cudaMalloc(&V2, sizeof(v)) || cudaMalloc(&nrm, sizeof(q)) ||
      cudaMalloc(&J, N * N * 4) || cudaMalloc(&stat, CL_MAX * 8 * 4) || cudaMalloc(&st, 256) || cudaMalloc(&out, 4)) return 3;
  cudaMemset(st, 0, 256);
  cudaMemcpy(W, w, sizeof(w), cudaMemcpyHostToDevice);
  cudaMemcpy(V, v, sizeof(v), cudaMemcpyHostToDevice);
  cudaMemcpy(nrm, q, sizeof(q), cudaMemcpyHostToDevice);
  if (cudaFuncSetAttribute(run, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM)) return 4;
  run<<<1, 512, SMEM>>>(W, V, V2, J, nrm, stat, st, 1e-26f, out);
  if (cudaMemcpy(&r, out, 4, cudaMemcpyDeviceToHost)) return 5;
  cudaMemcpy(w, W, sizeof(w), cudaMemcpyDeviceToHost);
  cudaMemcpy(v, V, sizeof(v), cudaMemcpyDeviceToHost);
  f = fopen(argv[2], "wb");
  fwrite(w, sizeof(w), 1, f);
  fwrite(v, sizeof(v), 1, f);
  fclose(f);
  printf("%%s\n", r == RF_DONE ? "done" : r == RF_SWEEPS ? "sweeps" : "dead");
  return 0;
}
""" % (N, LEN)


@pytest.fixture(scope="module")
def polish(tmp_path_factory):
    d = tmp_path_factory.mktemp("polish")
    src, exe = d / "polish.cu", d / "polish"
    src.write_text(PROGRAM)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    r = subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(W, V):
        np.concatenate([W.T.ravel(), V.T.ravel()]).tofile(d / "in")
        r = subprocess.run([str(exe), str(d / "in"), str(d / "out")], capture_output=True, text=True)
        assert r.returncode == 0, r.returncode
        o = np.fromfile(d / "out")
        return r.stdout.strip(), o[:N * LEN].reshape(N, LEN).T, o[N * LEN:].reshape(N, N).T

    return run


def columns(cosine, seed):
    """LEN x N columns over three decades whose pairs have about this cosine, and an orthogonal V."""
    rng = np.random.default_rng(seed)
    q = np.linalg.qr(rng.standard_normal((LEN, N + 1)))[0]
    w = np.sqrt(1 - cosine) * q[:, :N] + np.sqrt(cosine) * q[:, N:]
    return w * 10.0 ** (-3.0 * np.arange(N) / N), np.linalg.qr(rng.standard_normal((N, N)))[0]


@pytest.mark.parametrize("cosine,says", [(1e-10, "done"), (1e-5, "done"), (0.02, "sweeps"), (0.9, "sweeps")])
def test_polish_reports_what_it_reached(polish, cosine, says):
    W, V = columns(cosine, 7)
    got, w, v = polish(W, V)
    assert got == says
    if says == "done":
        g = w.T @ w
        d = np.sqrt(np.diag(g))
        c = g / np.outer(d, d) - np.eye(N)
        assert np.abs(c).max() <= 1.01e-13                       # the tolerance it is given, and the check's own rounding
        # second order in the cosines, 24 of them, and the FP32 products of what is taken off
        assert np.abs(w @ v.T - W @ V.T).max() <= N * cosine ** 2 + 24 * 6e-8 * cosine + 1e-15
    else:
        assert np.array_equal(w, W) and np.array_equal(v, V)
