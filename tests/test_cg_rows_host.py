"""The index arithmetic of the conjugate-gradient engine over all SMs, compiled
from its header with the host compiler (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1211_1581_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

HEAD = r"""
#include "cg_rows.h"
#include <climits>
#include <cstdio>
#include <vector>
using namespace mxm;
static int fails = 0;
#define CHECK(c) do { if (!(c)) { std::printf("FAIL %s line %d\n", #c, __LINE__); ++fails; } } while (0)
"""
TAIL = r"""
int main() {
  check();
  std::printf("%s %d\n", fails ? "FAILED" : "ok", fails);
  return fails ? 1 : 0;
}
"""


def run(tmp_path, body):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("host compiler or CUDA headers missing")
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(HEAD + body + TAIL)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover",
                    f"-I{CSRC}", f"-I{os.path.join(ROOT, 'include')}", f"-I{CUDA_INC}", str(src),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr


def test_rows_at_the_largest_count_of_values(tmp_path):
    """Every lane reads its own values of its row and no other, each once, for
    rows that end at or near INT32_MAX and however long the lane goes on
    beside a longer row of its warp."""
    run(tmp_path, r"""
void check() {
  const int kBatch = 8, ends[] = {INT_MAX, INT_MAX - 1, INT_MAX - 100, INT_MAX - 224, 70000, 100};
  for (int end : ends)
    for (int G = 1; G <= 32; G *= 2)
      for (int len : {0, 1, 7, 31, 32, 33, 100}) {
        const int begin = end - len;
        std::vector<int> seen(len, 0);
        for (int sub = 0; sub < G; ++sub) {
          RowWalk w = row_walk(begin, end, sub);
          int own = 0;
          for (int m = w.count(G) + 40 * kBatch; m > 0; m -= kBatch) {  // a longer row beside it
            for (int u = 0; u < kBatch; ++u)
              if (w.has(u * G)) {
                const long long at = static_cast<long long>(w.at) + u * G;
                CHECK(at >= begin && at < end && (at - begin) % G == sub);
                if (at >= begin && at < end) seen[at - begin]++;
                ++own;
              }
            w.advance(kBatch * G);
          }
          CHECK(own == (len > sub ? (len - sub - 1) / G + 1 : 0));
        }
        for (int v : seen) CHECK(v == 1);
      }
  // one row of all the values
  RowWalk w = row_walk(0, INT_MAX, 31);
  CHECK(w.count(32) == (INT_MAX - 32) / 32 + 1 && w.count(1) == INT_MAX - 31);
}
""")
