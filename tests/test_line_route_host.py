"""Host side of the short-line launch (no GPU): the shares of a cluster's CTAs cover a line of every
size within a tile, and a grid takes that launch only where the device reports room for the
cluster.  Compiled with nvcc and run on the host."""
import subprocess

import pytest

PROGRAM = r"""
#include <cstdio>
#include "tenom_internal.h"
#include "tenom_line.cuh"
using namespace tenom;

int main() {
  int bad = 0;
  for (int K = 6; K <= 8; K += 2) {
    for (int n = 1; n <= line_cells_max(K); ++n) {
      const int C = line_ctas(n), share = (n + C - 1) / C;
      if (C < 1 || C > LINE_CLUSTER || share * C < n || share + 1 + K - 1 > LINE_TILE) ++bad;
      if (!use_line(3, n, K, 1) || use_line(3, n, K, 0) || use_line(4, n, K, 1)) ++bad;
    }
    if (use_line(3, line_cells_max(K) + 1, K, 1)) ++bad;
  }
  std::printf("%d failing\n", bad);
  return bad ? 1 : 0;
}
"""


def test_line_shares_and_route(tmp_path):
    from paper_2010_13289_gb300 import build as B
    src, exe = tmp_path / "line_route.cu", tmp_path / "line_route"
    src.write_text(PROGRAM)
    r = subprocess.run([B.nvcc()] + B.ARCH + ["-std=c++17", "-O1", "-I", B.INCLUDE, "-I", B.CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail("nvcc failed:\n" + r.stderr[-3000:])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
