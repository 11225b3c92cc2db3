"""Work area of the cluster's FP64 centre SVDs, on the CPU: for every cluster size and every
shape, whatever way svd64_path takes it, all that the kernel places in the work area
ends within it, the staged rows of V and X included (the sweeps read them when they
finish what a refinement started)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_07615_gb300", "csrc")

PROGRAM = r"""
#include "rows_layout.cuh"
using namespace tn;

static long bad = 0;
static void check(bool ok, const char* what, int P, int ncol, int len, int eb) {
  if (!ok && bad++ < 20) printf("%s: P %d, %d x %d, %d bytes\n", what, P, ncol, len, eb);
}

int main() {
  long refined[2] = {0, 0};
  for (int eb = 4; eb <= 8; eb += 4)
    for (int P = 2; P <= 16; ++P)
      for (int ncol = 1; ncol <= 512; ++ncol)
        for (int len = ncol; len <= 1024; len += len < 300 ? 1 : 7) {
          const Svd64Path p = svd64_path(ncol, len, P, eb, true);
          if (!p.solo && !p.rows) continue;
          const int Pe = p.solo ? 1 : P;
          const int start = p.wide ? SW_WIDE : p.reg ? 0 : p.plain || eb == 8 ? SW_PLAIN : SW_SCRATCH;
          const RowsLayout R = rows_layout(ncol, len, Pe, rows_stage(eb, start));
          check(R.total <= (size_t)SM_WORK, "work area", P, ncol, len, eb);
          if (start == SW_PLAIN) continue;
          // W = X V: kc rows of V of ncol columns, kc rows of X of the CTA's lw entries
          check(R.st >= R.xb && R.xs >= R.st + (size_t)ncol * R.kc * 8, "staged V", P, ncol, len, eb);
          check(R.xs + (size_t)R.lw * R.kc * 8 <= R.sig, "staged X", P, ncol, len, eb);
          if (start == SW_SCRATCH) check(R.st >= R.gb + (size_t)ncol * R.lv * 8, "Newton-Schulz", P, ncol, len, eb);
          if (p.reg || p.wide) {
            check(rf_bytes(ncol, len, P) <= (size_t)SM_WORK, "refinement", P, ncol, len, eb);
            ++refined[eb == 8];
          }
          if (p.reg) check(2 * jacobi_reg_log_sweep(ncol) * 8 <= (size_t)SM_WORK, "log", P, ncol, len, eb);
          if (p.wide) check(jacobi_wide_smem(jacobi_wide_ldw(len)) <= (size_t)SM_WORK, "wide", P, ncol, len, eb);
        }
  printf("refined %ld %ld\n", refined[0], refined[1]);
  return bad ? 1 : refined[0] && refined[1] ? 0 : 2;
}
"""


def test_work_area_of_every_shape(tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "layout.cu", tmp_path / "layout"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
