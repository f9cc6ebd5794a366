// cg_rows.h -- how the conjugate-gradient engine over all SMs (cg_grid.cu)
// goes through the rows of a CSR matrix: index arithmetic alone, for the host
// as well as the device.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "mxm_internal.h"

namespace mxm {

// A lane's way through the values [begin, end) of a row, 0 <= begin <= end <=
// INT32_MAX: it takes begin + sub, then every G-th, G up to 32.  A lane whose row
// has ended goes on beside a longer row of its warp, up to end + the longest row
// + kWalkAhead: with more than kNarrowValues values that can pass INT32_MAX, and
// a 32-bit position would come out below the arrays, so Pos is 64 bits there.
// (64 bits for all: 1.4 million rows of 9 3315 us for 30 steps instead of 3190,
// 800,000 1340 instead of 1335.)
constexpr int32_t kWalkAhead = 256;  // 8 values of each of 32 lanes at a time
constexpr int32_t kNarrowValues = (1 << 30) - kWalkAhead;
template <typename Pos>
struct RowWalk {
  Pos at, end;
  __host__ __device__ bool has(int32_t offset) const { return at + offset < end; }
  __host__ __device__ void advance(int32_t step) { at += step; }
  // values that are the lane's own
  __host__ __device__ int32_t count(int32_t G) const {
    return at < end ? static_cast<int32_t>((end - at + G - 1) / G) : 0;
  }
};
template <typename Pos>
__host__ __device__ inline RowWalk<Pos> row_walk(int32_t begin, int32_t end, int32_t sub) {
  return RowWalk<Pos>{static_cast<Pos>(begin) + sub, end};
}

// Rows are shared out over kCgBlocks blocks (one per SM of a 152-SM GPU, a
// constant: the rounding of a solve does not depend on the device): share s
// takes rows [begin of s, begin of s + 1).
//
// By number where the values come out even.
constexpr int kCgBlocks = 152;
__host__ __device__ inline int64_t share_by_rows(int64_t n, int s) { return n * s / kCgBlocks; }

// Whether a share by number holds so many values that the shares are taken by
// work instead: more than twice the mean, and kShareSlack (four values a thread)
// beyond that, so that the chance differences of short shares do not count.
constexpr int64_t kShareSlack = 4096;
__host__ __device__ inline bool share_too_long(int64_t values, int64_t nnz) {
  return values > 2 * (nnz / kCgBlocks) + kShareSlack;
}

// By work: the row pointer plus kRowWork a row grows from 0 to the whole work; the
// share begins at the first row at or past s parts of it.  A row counts as one
// value: a lane's strided loads and gathers cost far more than the row's part of
// the dot products and vector updates (10^6 rows, the first tenth of 41 values,
// the rest of 5: 112 us a step; counted as two 117, as five 133; by number 233).
// Row pointers that are not in order give some other cut; the cuts still never
// decrease with s (each step of the search goes right for every larger s).
constexpr int64_t kRowWork = 1;
__host__ __device__ inline int64_t share_by_work(const int32_t* rowp, int64_t n, int64_t nnz,
                                                 int s) {
  if (s <= 0) return 0;
  if (s >= kCgBlocks) return n;
  const int64_t want = (nnz + kRowWork * n) * s / kCgBlocks;  // < 2^42 before the division
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (rowp[mid] + kRowWork * mid < want) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Rows longer than row_limit are not left to the G lanes that a row has by the
// mean length: a warp takes each, and above block_limit a whole block.  Four
// times the mean is no longer even; 256 values a lane take 32 rounds of eight
// loads, some 40 us, about a whole step.  A warp goes through block_limit values
// in 64 rounds.
__host__ __device__ inline int32_t row_limit(int64_t n, int64_t nnz, int G) {
  const int64_t four = 4 * ((nnz + n - 1) / n), most = four > 256 * G ? four : 256 * G;
  return static_cast<int32_t>(most < INT32_MAX ? most : INT32_MAX);
}
__host__ __device__ inline int32_t block_limit(int32_t row_limit) {
  const int64_t most = row_limit > 2048 ? 8 * static_cast<int64_t>(row_limit) : 16384;
  return static_cast<int32_t>(most < INT32_MAX ? most : INT32_MAX);
}

// How long a block waits for the others at a barrier.  The wait is for their
// work, most of all for a block that holds one row of nearly all the values: 0.3
// ns a value by a whole block, 0.8 by lanes that each have few rows.  So the limit
// grows with the number of values, five times what they may take (2^31 values:
// 10.6 s).
__host__ __device__ inline uint64_t cg_wait_limit_ns(int64_t nnz) {
  return kWaitLimitNs + 4 * static_cast<uint64_t>(nnz);
}

}  // namespace mxm
