"""CPU check of the columns at which the pipelined update on masked lattices looks
(mask_look.cuh, compiled here for the host): every one lies inside the row, for
every lane of every warp of every tile, and together the looks of a warp that has
nodes cover the neighbourhood of each.  Nothing here runs on a GPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2602_06686_gb300", "csrc")

MAIN = r"""
#define __host__
#define __device__
#include <cstdio>
#include <vector>
#include "mask_look.cuh"
using namespace lbm;

// layout 0: one node per thread (x0 + t); 1: the split pair (x0 + t, x0 + t + X/2);
// 2: the adjacent pair (x0 + 2t, x0 + 2t + 1), whose nodes look left and right
static int check(int nx, int X, int layout) {
  int bad = 0;
  std::vector<char> seen(nx);
  for (int x0 = 0; x0 < nx; x0 += X) {
    const int threads = layout == 0 ? X : X / 2;
    for (int w = 0; w < threads; w += 32) {
      seen.assign(nx, 0);
      std::vector<int> nodes;
      for (int l = 0; l < 32; ++l)
        for (int k = 0; k < (layout == 0 ? 1 : 2); ++k) {
          const int t = w + l;
          const int x = x0 + (layout == 2 ? 2 * t + k : t + k * (X / 2));
          const int as = layout == 2 ? 31 * k : l;  // the lane that mask_near is given
          for (int c : {mask_column(x, nx), mask_column_beside(x, nx, as)}) {
            if (c < 0 || c >= nx) ++bad;
            else seen[c] = 1;
          }
          if (x < nx && x < x0 + X) nodes.push_back(x);
        }
      for (int x : nodes)
        if (!seen[x] || !seen[(x + 1) % nx] || !seen[(x + nx - 1) % nx]) ++bad;
    }
  }
  return bad;
}

int main() {
  for (int X : {128, 256, 384, 512})
    for (int layout = 0; layout < 3; ++layout)
      for (int nx = 4; nx <= 1100; ++nx)
        if (int b = check(nx, X, layout)) {
          std::printf("nx %d tile %d layout %d: %d\n", nx, X, layout, b);
          return 1;
        }
  return 0;
}
"""


def test_mask_columns_stay_in_the_row_and_cover_every_node(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "columns.cpp"
    src.write_text(MAIN)
    exe = tmp_path / "columns"
    subprocess.run([cxx, "-O2", "-std=c++17", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
