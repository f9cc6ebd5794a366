"""What bench.py divides by its times, against the library: the number of digit
products at the benchmark's size, from the rule in the library's header (host
compiler, no GPU), and the sources whose hash ties a profile to a kernel."""
import os
import re
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1211_1581_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"
sys.path.insert(0, ROOT)

PROGRAM = r"""
#include "mxm_internal.h"
#include <cstdio>
using namespace mxm;
int main() {  // beta, balanced, slices, products
  for (int kind = 0; kind < 3; ++kind)
    for (int S = 1; S <= (kind == 2 ? kOzMaxSlicesRn8 : kOzMaxSlices); ++S) {
      const OzakiDims d = ozaki_dims(8192, 8192, 8192, S, kind == 0 ? 7 : 8, kind == 2);
      const int n = kara_chosen(d) ? (S - 1) + kara_pairs(S) + 2 : S * (S + 1) / 2;
      std::printf("%d %d %d %d\n", d.beta, d.rn, S, n);
    }
}
"""


def test_digit_products(tmp_path):
    import bench
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("host compiler or CUDA headers missing")
    src, exe = tmp_path / "count.cpp", tmp_path / "count"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", f"-I{CSRC}", f"-I{os.path.join(ROOT, 'include')}",
                    f"-I{CUDA_INC}", str(src), "-o", str(exe)], check=True)
    rows = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")
    rows = [tuple(map(int, r.split())) for r in rows if r]
    assert (8, 0, 6, 15) in rows and (7, 0, 7, 19) in rows
    for beta, _, S, products in rows:
        assert bench.digit_products(S, beta) == products, (beta, S)


def test_profiled_sources_are_all_of_the_kernels():
    import bench
    names = {os.path.basename(p) for p in bench.PRODUCT_SOURCES}
    todo = ["ozaki_kara.cu"]
    while todo:
        name = todo.pop()
        assert name in names
        with open(os.path.join(CSRC, name)) as fh:
            own = re.findall(r'#include "([^"]+)"', fh.read())
        todo += [o for o in own if os.path.exists(os.path.join(CSRC, o)) and o not in todo]
