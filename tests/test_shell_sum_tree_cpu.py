"""The lane sums of the P(k) shells, run on the host from the kernels' header: five FP32 additions
deep for every rotation, so within 5 x 2^-24 of the exact sum of positive values.  A chain loses all
31 small values beside a large one (31 x 2^-24)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include "passes.cuh"
int main() {
  for (int big = 0; big < 32; ++big) {
    float row[32];
    double want = 0.0;
    for (int i = 0; i < 32; ++i) want += row[i] = i == big ? 1.0f : 0x1p-24f;
    for (int rot = 0; rot < 32; ++rot) {
      const double got = lpt2::tree_sum<32>(row, rot);
      if (std::fabs(got - want) > 5 * 0x1p-24 * want) return std::printf("%d %d %.9g\n", big, rot, got), 1;
    }
  }
  return 0;
}
"""


def test_lane_sums_are_a_tree(tmp_path):
    from paper_1909_06282_gb300 import build as B

    src, exe = tmp_path / "tree.cu", tmp_path / "tree"
    src.write_text(SOURCE)
    cmd = [B.nvcc(), *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-I", os.path.join(ROOT, "include"),
           str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
