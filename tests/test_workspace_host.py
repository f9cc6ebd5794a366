"""Which buffer a call gets, and what that costs, with a fake allocator: the
library's rules compiled with the host compiler (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1211_1581_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

PROGRAM = r"""
#include "workspace.h"
#include <cstdio>
#include <map>
using namespace mxm;
static int fails = 0;
#define CHECK(c) do { if (!(c)) { std::printf("FAIL %s line %d\n", #c, __LINE__); ++fails; } } while (0)
constexpr size_t MB = size_t(2) << 20;  // the granularity of the library's buffers
struct Fake {
  size_t memory, largest = SIZE_MAX;  // in all; of one piece
  bool capture = false;
  int syncs = 0, tries = 0, frees = 0, next = 1;
  std::map<void*, size_t> held;
  size_t used() const { size_t n = 0; for (auto& h : held) n += h.second; return n; }
  bool capturing() const { return capture; }
  bool synchronize() { ++syncs; return true; }
  bool allocate(void** p, size_t n) {
    ++tries;
    *p = nullptr;
    if (n > largest || used() + n > memory) return false;
    *p = reinterpret_cast<void*>(static_cast<uintptr_t>(next++) << 21);
    held[*p] = n;
    return true;
  }
  void release(void* p) { ++frees; CHECK(held.erase(p) == 1); }
  bool available(size_t* n) { *n = memory - used(); return true; }
  int calls() const { return syncs + tries + frees; }
};
int main() {
  {  // room for both: the larger one, the old one given back after a synchronisation
    Fake a{1000 * MB};
    Workspace w;
    CHECK(workspace_need(w, 40 * MB, a) == MXM_OK && w.bytes >= 40 * MB && a.syncs == 0);
    CHECK(workspace_want(w, 80 * MB, 40 * MB, a) && w.bytes >= 80 * MB);
    CHECK(a.syncs == 1 && a.frees == 1 && a.held.size() == 1 && a.held.count(w.base) == 1);
    const int before = a.calls();
    CHECK(workspace_want(w, 80 * MB, 40 * MB, a) && a.calls() == before);
  }
  {  // not to be had: the buffer stays where it is, and is not asked about again
    Fake a{100 * MB};
    Workspace w;
    CHECK(workspace_need(w, 40 * MB, a) == MXM_OK);
    void* const base = w.base;
    CHECK(!workspace_want(w, 110 * MB, 40 * MB, a));
    CHECK(w.base == base && w.bytes >= 40 * MB && a.syncs == 0 && a.frees == 0);
    const int before = a.calls();
    for (int i = 0; i < 100; ++i) {
      CHECK(!workspace_want(w, 110 * MB, 40 * MB, a));
      CHECK(workspace_need(w, 40 * MB, a) == MXM_OK && w.base == base);
    }
    CHECK(!workspace_want(w, 200 * MB, 40 * MB, a) && a.calls() == before);
    CHECK(workspace_want(w, 50 * MB, 40 * MB, a) && a.held.size() == 1);  // a smaller one is
  }
  {  // the two do not fit together, the larger one alone does
    Fake a{100 * MB};
    Workspace w;
    CHECK(workspace_need(w, 40 * MB, a) == MXM_OK);
    CHECK(workspace_want(w, 80 * MB, 40 * MB, a) && w.bytes >= 80 * MB && a.held.size() == 1);
  }
  {  // refused all the same: the size that was there comes back
    Fake a{100 * MB, 60 * MB};
    Workspace w;
    CHECK(workspace_need(w, 40 * MB, a) == MXM_OK);
    CHECK(!workspace_want(w, 80 * MB, 40 * MB, a));
    CHECK(w.base != nullptr && w.bytes >= 40 * MB && a.held.size() == 1 && a.held.count(w.base));
    const int before = a.calls();
    CHECK(!workspace_want(w, 80 * MB, 40 * MB, a) && workspace_need(w, 40 * MB, a) == MXM_OK);
    CHECK(a.calls() == before);
  }
  {  // a buffer too small for the call at all
    Fake a{100 * MB};
    Workspace w;
    CHECK(workspace_need(w, 10 * MB, a) == MXM_OK);
    CHECK(!workspace_want(w, 110 * MB, 40 * MB, a));
    CHECK(workspace_need(w, 40 * MB, a) == MXM_OK && a.held.size() == 1);
    const int before = a.calls();
    CHECK(!workspace_want(w, 110 * MB, 40 * MB, a) && workspace_need(w, 40 * MB, a) == MXM_OK);
    CHECK(a.calls() == before);
    CHECK(workspace_need(w, 200 * MB, a) == MXM_ERR_CUDA && w.base == nullptr && w.bytes == 0);
  }
  {  // a capture allocates nothing, a caller's buffer is never given back
    Fake a{1000 * MB};
    Workspace w;
    CHECK(workspace_need(w, 40 * MB, a) == MXM_OK);
    a.capture = true;
    const int before = a.calls();
    CHECK(!workspace_want(w, 80 * MB, 40 * MB, a) && w.refused == SIZE_MAX);
    CHECK(workspace_need(w, 40 * MB, a) == MXM_OK);
    CHECK(workspace_need(w, 80 * MB, a) == MXM_ERR_NO_WORKSPACE && a.calls() == before);
    a.capture = false;
    Workspace c;
    c.base = &c;
    c.bytes = 50 * MB;
    c.owned = false;
    CHECK(!workspace_want(c, 80 * MB, 40 * MB, a) && workspace_need(c, 40 * MB, a) == MXM_OK);
    CHECK(workspace_need(c, 80 * MB, a) == MXM_ERR_WORKSPACE_TOO_SMALL && a.calls() == before);
  }
  std::printf("%s %d\n", fails ? "FAILED" : "ok", fails);
  return fails ? 1 : 0;
}
"""


def test_buffers_of_a_call(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("host compiler or CUDA headers missing")
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", f"-I{CSRC}", f"-I{os.path.join(ROOT, 'include')}",
                    f"-I{CUDA_INC}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
