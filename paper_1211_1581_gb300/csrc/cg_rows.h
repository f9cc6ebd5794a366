// cg_rows.h -- how the conjugate-gradient engine over all SMs (cg_grid.cu)
// goes through the rows of a CSR matrix: index arithmetic alone, for the host
// as well as the device.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace mxm {

// A lane's way through the values [begin, end) of a row, 0 <= begin <= end <=
// INT32_MAX: it takes begin + sub, then every G-th.  In 64 bits: a lane whose row
// has ended goes on beside a longer row of its warp, and past INT32_MAX a 32-bit
// position would come out below the arrays.  (Counting the values left in 32
// bits instead is exact too, but slower: 10^6 rows of 7 1077 us for 30 steps,
// 300,000 of 21 945 us, against 1050 and 912.)
struct RowWalk {
  int64_t at, end;
  __host__ __device__ bool has(int32_t offset) const { return at + offset < end; }
  __host__ __device__ void advance(int32_t step) { at += step; }
  // values that are the lane's own
  __host__ __device__ int32_t count(int32_t G) const {
    return at < end ? static_cast<int32_t>((end - at + G - 1) / G) : 0;
  }
};
__host__ __device__ inline RowWalk row_walk(int32_t begin, int32_t end, int32_t sub) {
  return RowWalk{static_cast<int64_t>(begin) + sub, end};
}

}  // namespace mxm
