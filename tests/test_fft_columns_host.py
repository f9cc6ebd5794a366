"""How many columns a CTA of a transform's pass takes, from the library's header
with the host compiler (no GPU): waves as full as they can be, and among equally
full ones as many CTAs as keep every thread at work."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1211_1581_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

PROGRAM = r"""
#include "mxm_internal.h"
#include <cstdio>
using namespace mxm;
static int fails = 0;
#define CHECK(c) do { if (!(c)) { std::printf("FAIL %s line %d: %d of %lld, %d SMs\n", #c, __LINE__, bits, cols, sms); ++fails; } } while (0)
static double fill(long long cols, int cb, int sms) {
  const long long b = cols >> cb;
  return static_cast<double>(b) / static_cast<double>((b + sms - 1) / sms * sms);
}
int main() {
  for (int sms : {152, 148, 76, 20})
    for (int p = 2; p <= 22; ++p)
      for (int pass = 0; pass < 2; ++pass) {
        const int b1 = (p + 1) / 2, bits = pass ? p - b1 : b1;
        const long long cols = 1ll << (p - bits);
        const int cb = fft_column_bits(bits, cols, sms);
        CHECK(cb >= 0 && cb <= 3 && (cols >> cb) >= 1);
        CHECK((((1ll << cb) + 1) << bits) * 16 <= 96 * 1024 || cb == 0);
        for (int o = 0; o <= 3; ++o) {  // no other count is fuller where none is full enough
          if (cols < (1ll << o) || (((1ll << o) + 1) << bits) * 16 > 96 * 1024) continue;
          if (fill(cols, cb, sms) < 0.9) CHECK(fill(cols, o, sms) <= fill(cols, cb, sms));
          // nor as full with more CTAs that still have a butterfly a thread
          if (fill(cols, cb, sms) < 0.9 && o < cb && (1ll << (o + bits)) >= 4 * kFftThreads)
            CHECK(fill(cols, o, sms) < fill(cols, cb, sms));
        }
      }
  int bits = 10, sms = 152;
  long long cols = 512;
  CHECK(fft_column_bits(10, 512, 152) == 0);  // 2^19, first pass: 512 CTAs, not 128
  bits = 9;
  CHECK(fft_column_bits(9, 512, 152) == 1);   // 2^18: 256 CTAs
  std::printf("%s %d\n", fails ? "FAILED" : "ok", fails);
  return fails ? 1 : 0;
}
"""


def test_columns_per_cta(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("host compiler or CUDA headers missing")
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", f"-I{CSRC}", f"-I{os.path.join(ROOT, 'include')}",
                    f"-I{CUDA_INC}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
