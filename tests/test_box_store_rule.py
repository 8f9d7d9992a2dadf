"""The rule that lets the fp32 GEMM epilogue write its result by box stores (host code, no GPU): a
warp fills its two staging buffers in turn, beginning with the first in every tile, and before a
chunk waits until at most one store is still reading.  That is enough only if no chunk takes the buffer
of the chunk right before it, across tiles too."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_06411_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "kernels.h"
int main() {
  for (int tile : {128, 256})
    for (int n = 4; n <= 1024; n += 4) {
      mapk::GemmDesc d{};
      d.epi = mapk::EPI_F32; d.M = 300; d.N = n; d.K = 64; d.batch = 1;
      int reading = -1, clash = 0;                       // buffer that the last store may still read
      for (int t = 0; t < 3; ++t)                        // tiles of one CTA, the last column tile each time
        for (int ch = 0, c0 = (n - 1) / tile * tile; ch < tile / 32 && c0 + 32 * ch < n; ++ch) {
          clash |= (ch & 1) == reading;
          reading = ch & 1;
        }
      if (mapk::f32_box_store(d)) std::printf("%d %d %d\n", tile, n, clash);
    }
}
"""


def test_box_stores_never_refill_a_buffer_that_is_being_read(tmp_path):
    gxx = shutil.which("g++")
    cuda = "/usr/local/cuda/include"
    if not gxx or not os.path.isdir(cuda):
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "rule.cc"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, "-I", cuda, str(src), "-o", str(tmp_path / "rule")], check=True)
    rows = [tuple(map(int, line.split())) for line in
            subprocess.run([str(tmp_path / "rule")], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert [r for r in rows if r[2]] == []
    assert {n for _, n, _ in rows} >= set(range(64, 1025, 64))      # widths of the library's own calls
