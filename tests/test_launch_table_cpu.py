"""CPU check of the table in which the launchers keep a kernel's shared-memory opt-in and
occupancy (launch_table.h, compiled here for the host with fakes of the two runtime calls):
both are asked for once per device and ring depth, errors are not kept, and host threads
may ask at the same time.  Nothing here runs on a GPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2602_06686_gb300", "csrc")
CUDA = "/usr/local/cuda/include"

MAIN = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "launch_table.h"
using namespace lbm;
#define CHECK(c) if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; }

int main() {
  static LaunchTable t;
  int set[32] = {}, asked[32] = {}, n = 0;
  const auto get = [&](int dev, int depth, cudaError_t set_rc, int value) {
    return t.get(dev, depth, [&] { ++set[dev]; return set_rc; },
                 [&](int* v) { ++asked[dev]; *v = value; return cudaSuccess; }, &n);
  };
  // an error is returned and not kept
  CHECK(get(0, 3, cudaErrorInvalidValue, 4) == cudaErrorInvalidValue && asked[0] == 0);
  CHECK(get(0, 3, cudaSuccess, 0) == cudaErrorInvalidConfiguration);
  CHECK(get(0, 3, cudaSuccess, 4) == cudaSuccess && n == 4);
  const int s0 = set[0], a0 = asked[0];
  for (int k = 0; k < 5; ++k) CHECK(get(0, 3, cudaSuccess, 7) == cudaSuccess && n == 4);
  CHECK(set[0] == s0 && asked[0] == a0);  // kept
  CHECK(get(0, 2, cudaSuccess, 6) == cudaSuccess && n == 6);  // another depth is another entry
  CHECK(get(1, 3, cudaSuccess, 5) == cudaSuccess && n == 5 && set[1] == 1);  // another device opts in itself
  CHECK(get(0, 3, cudaSuccess, 9) == cudaSuccess && n == 4);
  // beyond the table: asked every time
  CHECK(get(20, 3, cudaSuccess, 2) == cudaSuccess && n == 2);
  CHECK(get(20, 3, cudaSuccess, 3) == cudaSuccess && n == 3 && set[20] == 2);
  // threads
  static LaunchTable u;
  std::vector<std::thread> th;
  std::vector<int> got(8 * 64);
  for (int k = 0; k < 8; ++k)
    th.emplace_back([&, k] {
      for (int r = 0; r < 64; ++r)
        u.get(r % 8, 2, [] { return cudaSuccess; }, [&](int* v) { *v = 1 + r % 8; return cudaSuccess; },
              &got[k * 64 + r]);
    });
  for (auto& x : th) x.join();
  for (int k = 0; k < 8; ++k)
    for (int r = 0; r < 64; ++r) CHECK(got[k * 64 + r] == 1 + r % 8);
  return 0;
}
"""


def test_launch_table_is_per_device_and_depth(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    src = tmp_path / "table.cpp"
    src.write_text(MAIN)
    exe = tmp_path / "table"
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", f"-I{CSRC}", f"-I{CUDA}", str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
