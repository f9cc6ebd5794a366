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
const int kBatch = 8;
template <typename Pos>
static void walks(const std::vector<int>& ends) {
  for (int end : ends)
    for (int G = 1; G <= 32; G *= 2)
      for (int len : {0, 1, 7, 31, 32, 33, 100}) {
        const int begin = end - len;
        std::vector<int> seen(len, 0);
        for (int sub = 0; sub < G; ++sub) {
          auto w = row_walk<Pos>(begin, end, sub);
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
}
void check() {
  walks<int64_t>({INT_MAX, INT_MAX - 1, INT_MAX - 100, INT_MAX - 224, 70000, 100});
  walks<int32_t>({kNarrowValues, kNarrowValues - 1, 70000, 100});
  // one row of all the values, and a lane of the last row beside it to its end
  auto w = row_walk<int64_t>(0, INT_MAX, 31);
  CHECK(w.count(32) == (INT_MAX - 32) / 32 + 1 && w.count(1) == INT_MAX - 31);
  for (int G = 1; G <= 32; G *= 2) {
    auto one = row_walk<int32_t>(0, kNarrowValues, 0);
    auto last = row_walk<int32_t>(kNarrowValues - 1, kNarrowValues, G - 1);
    for (int m = one.count(G); m > 0; m -= kBatch) {
      const bool mine = last.has(0) && last.at == kNarrowValues - 1;
      for (int u = 0; u < kBatch; ++u) CHECK(last.has(u * G) == (mine && u == 0));
      last.advance(kBatch * G);
    }
  }
}
""")


def test_shares_of_uneven_rows(tmp_path):
    """The cut by work covers every row once and gives no share more than its
    part of the work and one row; it is taken where neighbouring rows hold most
    of the values and not for rows of one length, or of chance lengths.  Row
    pointers out of order still give cuts that never decrease."""
    run(tmp_path, r"""
static std::vector<int> pointers(const std::vector<int>& len) {
  std::vector<int> p(1, 0);
  for (int l : len) p.push_back(p.back() + l);
  return p;
}
static bool by_work(const std::vector<int>& p) {
  const long long n = static_cast<long long>(p.size()) - 1;
  for (int s = 0; s < kCgBlocks; ++s)
    if (share_too_long(p[share_by_rows(n, s + 1)] - p[share_by_rows(n, s)], p[n])) return true;
  return false;
}
void check() {
  unsigned long long seed = 1;
  auto rnd = [&](int m) { return static_cast<int>((seed = seed * 6364136223846793005ull + 1442695040888963407ull) >> 33) % m; };
  std::vector<std::vector<int>> uneven, even;
  std::vector<int> l(200000, 3);
  for (int i = 0; i < 1316; ++i) l[i] = 658;
  uneven.push_back(l);
  l.assign(160001, 2); l[80000] = 160001;
  uneven.push_back(l);
  l.assign(5000, 2); l[4999] = 5000;
  uneven.push_back(l);
  l.assign(100, 0); l[7] = 3000000;
  uneven.push_back(l);
  l.assign(1, 1000000);
  uneven.push_back(l);
  for (int n : {1, 100, 151, 152, 153, 12288, 200000}) {
    l.assign(n, 7);
    even.push_back(l);
    for (int& v : l) v = rnd(33);
    even.push_back(l);
    l.assign(n, 0);
    even.push_back(l);
  }
  for (const auto& len : uneven) CHECK(by_work(pointers(len)));
  for (const auto& len : even) CHECK(!by_work(pointers(len)));
  uneven.insert(uneven.end(), even.begin(), even.end());
  for (const auto& len : uneven) {
    const std::vector<int> p = pointers(len);
    const long long n = static_cast<long long>(len.size()), nnz = p[n];
    const long long part = (nnz + kRowWork * n) / kCgBlocks + 1;
    CHECK(share_by_work(p.data(), n, nnz, 0) == 0 && share_by_work(p.data(), n, nnz, kCgBlocks) == n);
    for (int s = 0; s < kCgBlocks; ++s) {
      const long long lo = share_by_work(p.data(), n, nnz, s), hi = share_by_work(p.data(), n, nnz, s + 1);
      CHECK(lo <= hi && hi <= n);
      CHECK(lo == hi || (p[hi - 1] + kRowWork * (hi - 1)) - (p[lo] + kRowWork * lo) <= part);
    }
  }
  for (int r = 0; r < 200; ++r) {  // anything at all in the row pointers
    const int n = 1 + rnd(3000);
    std::vector<int> p(n + 1);
    for (int& v : p) v = (rnd(2) ? 1 : -1) * rnd(INT_MAX);
    for (int s = 0; s < kCgBlocks; ++s) {
      const long long lo = share_by_work(p.data(), n, 100000, s), hi = share_by_work(p.data(), n, 100000, s + 1);
      CHECK(0 <= lo && lo <= hi && hi <= n);
    }
  }
}
""")


def test_limits_of_long_rows(tmp_path):
    """Rows up to four times the mean, and up to 256 values a lane, stay with
    their lanes; the limits do not overflow at the largest counts."""
    run(tmp_path, r"""
void check() {
  for (long long n : {1ll, 152ll, 5000ll, 160001ll, 1000000ll, 2147483647ll})
    for (long long nnz : {0ll, 1ll, 3 * n, 40 * n, 2147483647ll})
      for (int G = 1; G <= 32; G *= 2) {
        if (nnz > 2147483647ll) continue;
        const long long r = row_limit(n, nnz, G), b = block_limit(static_cast<int>(r));
        CHECK(r >= 256 * G && (r == INT_MAX || r >= 4 * (nnz / n)));
        CHECK(b >= 16384 && (b == INT_MAX || b >= 8 * r) && b >= r);
      }
  CHECK(row_limit(160001, 480001, 1) == 256 && block_limit(256) == 16384);
  CHECK(row_limit(1000, 2147483647, 32) == 4 * 2147484);
}
""")


def test_wait_limit_grows_with_the_values(tmp_path):
    """A block may hold a row of all the values: the wait for it allows ns for
    each beyond the usual limit, and stays bounded."""
    run(tmp_path, r"""
void check() {
  CHECK(cg_wait_limit_ns(0) == kWaitLimitNs);
  for (long long nnz : {1000ll, 60000000ll, 2147483647ll})
    CHECK(cg_wait_limit_ns(nnz) >= kWaitLimitNs + 4 * nnz && cg_wait_limit_ns(nnz) < 20000000000ull);
}
""")
