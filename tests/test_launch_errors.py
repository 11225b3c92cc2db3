"""A cluster launch that fails is reported by the function that launches it: on a machine
without a GPU every launch fails."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_07615_gb300", "csrc")

PROGRAM = r"""
#include "internal.cuh"
int main() {
  cudaError_t e = tn::launch_gram_eig(nullptr, nullptr, 64, nullptr, 32, 0.0, 64, nullptr, nullptr, 0);
  printf("%s\n", cudaGetErrorString(e));
  return e == cudaSuccess ? 1 : 0;
}
"""


def test_gram_eig_launch_error(tmp_path):
    import torch
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if torch.cuda.is_available() or not os.path.exists(nvcc):
        pytest.skip("needs nvcc and no GPU")
    from paper_2512_07615_gb300 import build
    lib = build.build()
    src, exe = tmp_path / "launch.cu", tmp_path / "launch"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-cudart", "shared", "-I", CSRC,
                        str(src), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
