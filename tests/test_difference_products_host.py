"""The host-side rules of the difference products, compiled from the library's
internal header with the host compiler (no GPU): the plane numbering, the
FP32 windows and the int32 bounds; and the identity itself, by brute force on
random digit vectors."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1211_1581_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

PROGRAM = r"""
#include "mxm_internal.h"
#include <cstdio>
#include <vector>
using namespace mxm;
static int fails = 0;
#define CHECK(c) do { if (!(c)) { std::printf("FAIL %s line %d\n", #c, __LINE__); ++fails; } } while (0)
int main() {
  for (int S = 3; S <= kKaraMaxSlices; ++S) {
    // every pair s < t, s + t <= S + 1, but (1, S), has a plane of its own
    std::vector<int> seen(kara_planes(S), 0);
    for (int s = 1; s <= S; ++s) seen[s - 1]++;
    for (int s = 1; s <= S; ++s)
      for (int t = s + 1; s + t <= S + 1; ++t) {
        if (s == 1 && t == S) continue;
        const int p = kara_pair_plane(S, s, t);
        CHECK(p >= S && p < kara_planes(S));
        if (p >= 0 && p < kara_planes(S)) seen[p]++;
      }
    for (int v : seen) CHECK(v == 1);
  }
  // windows stay within 2^24: truncated digits keep their bound, balanced
  // digits differ by up to 256
  OzakiDims d = ozaki_dims(1024, 1024, 1024, 7, 7);
  CHECK(kara_window_stages(d) * 128ll * 127 * 127 <= (1ll << 24));
  d = ozaki_dims(1024, 1024, 1024, 6, 8);
  CHECK(kara_window_stages(d) * 128ll * 255 * 255 <= (1ll << 24));
  d = ozaki_dims(1024, 1024, 1024, 6, 8, true);
  CHECK(kara_window_stages(d) >= 1 && kara_window_stages(d) * 128ll * 256 * 256 <= (1ll << 24));
  // the choice: two tile-rows and tile-columns, sums in int32, bounded memory
  CHECK(kara_chosen(ozaki_dims(129, 64, 129, 7, 7)));
  CHECK(!kara_chosen(ozaki_dims(128, 64, 1024, 7, 7)));
  CHECK(!kara_chosen(ozaki_dims(1024, 64, 128, 7, 7)));
  CHECK(kara_chosen(ozaki_dims(1024, 300, 100, 7, 7)));
  CHECK(!kara_chosen(ozaki_dims(32768, 1024, 64, 7, 7)));
  CHECK(!kara_chosen(ozaki_dims(1024, 1024, 1024, 2, 7)));
  CHECK(!kara_chosen(ozaki_dims(1024, 1024, 1024, 10, 7)));
  CHECK(kara_chosen(ozaki_dims(8192, 8192, 8192, 7, 7)));
  d = ozaki_dims(8192, 8192, 8192, 6, 8);  // D_g beyond int32: k in ranges within it
  CHECK(kara_chosen(d) && kara_min_ranges(d) == 2 && !ozaki_narrow(d));
  CHECK(7.0 * 255 * 255 * 128 * ((d.Kt + 1) / 2) < 2147483648.0);
  CHECK(kara_min_ranges(ozaki_dims(8192, 8192, 8192, 7, 7)) == 1);
  CHECK(kara_chosen(ozaki_dims(8192, 8192, 8192, 6, 8, true)));
  CHECK(!kara_chosen(ozaki_dims(65536, 16384, 65536, 7, 7)));   // memory
  std::printf("%s %d\n", fails ? "FAILED" : "ok", fails);
  return fails ? 1 : 0;
}
"""


def test_planes_windows_and_choice(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("host compiler or CUDA headers missing")
    src, exe = tmp_path / "kara_check.cpp", tmp_path / "kara_check"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", f"-I{CSRC}", f"-I{os.path.join(ROOT, 'include')}",
                    f"-I{CUDA_INC}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr


@pytest.mark.parametrize("S", range(3, 10))
def test_identity(S):
    """D_g from the squares and the difference products equals the sum of the
    digit products, in integers."""
    rng = np.random.default_rng(S)
    a = rng.integers(-127, 128, (S + 1, 50)).astype(object)
    b = rng.integers(-127, 128, (S + 1, 50)).astype(object)
    P = [0] + [int(a[s] @ b[s]) for s in range(1, S)]
    for g in range(2, S + 2):
        want = sum(int(a[s] @ b[g - s]) for s in range(1, g) if g - s <= S)
        got = sum(P[1:min(g, S)])
        for s in range(1, g):
            t = g - s
            if s >= t:
                break
            if (s, t) == (1, S):
                got += int(a[1] @ b[S]) + int(a[S] @ b[1]) - P[1]
            else:
                got += int((a[s] - a[t]) @ (b[t] - b[s]))
        assert got == want, g
