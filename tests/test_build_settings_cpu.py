"""The pass configurations under the library's build settings, checked on the host: a small program
made from the kernels' headers (no GPU is touched) evaluates the constants that the kernels are
instantiated with."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1909_06282_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include "passes.cuh"
using namespace lpt2;
int bad = 0;
void fail(const char* what, int n, int a, int b) { std::printf("%s N=%d %d %d\n", what, n, a, b); ++bad; }

// every twiddle that the stages of schedule V read is the one they mean
template <int N, int V> void twiddles(const char* pass) {
  for (int s = 1; s < Cfg<N, V>::NS; ++s) {
    const int ns = ns_before<N, V>(s), R = Cfg<N, V>::rad(s);
    for (int r = 1; r < R; ++r)
      for (int j = 0; j < ns; ++j)
        if (twiddle_exponent<N>(r * ns + j) != r * j * (N / (ns * R))) return fail(pass, N, s, r * ns + j);
  }
}
template <int N, int MODE> void x() {
  using C = XCfg<N, MODE>;
  twiddles<N, C::V>("x twiddles");
  // the sums over modes go by whole warps, a power of two of them in the shell sums
  const bool shells = MODE == X_PKP || MODE == X_PKI;
  if (shells || MODE == X_PK || MODE == X_ADJ_SOURCE) {
    const int nwarp = C::XT / 32;
    if (C::XT % 32 || nwarp < 1 || (shells && (nwarp & (nwarp - 1)))) fail("x warps", N, MODE, C::XT);
  }
}
template <int N, int KIND> void y() {
  twiddles<N, YCfg<N, KIND>::V>("y twiddles");
  twiddles<N, YCfg<N, KIND, 8>::V>("y twiddles");
  if constexpr (N >= 32) twiddles<N, YCfg<N, KIND, 16>::V>("y twiddles");
}
// the z passes' groups exist and fit on an SM (227 KB); named barriers are 0 .. 15
template <int N> void z() {
  using Q = ZGrp<N>;
  if (Q::SMEM > 232448) fail("z group memory", N, Q::SMEM, 0);
  if (Q::GT > 32 && Q::GROUPS > 15) fail("z group barriers", N, Q::GT, Q::GROUPS);
}
template <int N> void all() {
  z<N>();
  twiddles<N, 0>("z twiddles");
  y<N, Y_MULTI>(); y<N, Y_SUM>(); y<N, Y_ONE>();
  x<N, X_FWD>(); x<N, X_INV>(); x<N, X_MUL>(); x<N, X_DELTA>(); x<N, X_SOURCE>(); x<N, X_PK>(); x<N, X_PKP>();
  x<N, X_PKI>(); x<N, X_PKADJ>(); x<N, X_ADJ_SOURCE>(); x<N, X_ADJ_DELTA>();
}
int main() {
  all<16>(); all<32>(); all<64>(); all<96>(); all<128>(); all<192>(); all<256>(); all<512>(); all<1024>();
  return bad ? 1 : 0;
}
"""


@pytest.mark.parametrize("setting", ["", "-DLPT2_R512=8", "-DLPT2_W512=16", "-DLPT2_WSMALL=4", "-DLPT2_WSMALL=8",
                                     "-DLPT2_ZTHREADS=128", "-DLPT2_ZTHREADS=512"])
def test_pass_configurations(setting, tmp_path):
    from paper_1909_06282_gb300 import build as B

    src, exe = tmp_path / "settings.cu", tmp_path / "settings"
    src.write_text(SOURCE)
    cmd = [B.nvcc(), *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
           *setting.split(), str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
