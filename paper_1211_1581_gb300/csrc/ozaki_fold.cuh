// ozaki_fold.cuh -- what the slice GEMMs share: the walk over C tiles and the
// pieces of the FP64 recombination (step 4 of the method in ozaki.cu).
#pragma once
#include <cstdint>

#include "mxm_internal.h"
#include "ptx.cuh"

namespace mxm {

__device__ __forceinline__ void tile_coords(int64_t tile, int64_t Mt, int64_t Nt, int64_t G,
                                            int64_t& tm, int64_t& tn) {
  // groups of G tile-rows, column-major inside a group: CTAs working at the
  // same time share A tiles and B tiles in L2
  const int64_t per_group = G * Nt;
  const int64_t grp = tile / per_group;
  const int64_t first = grp * G;
  const int64_t gsz = (Mt - first) < G ? (Mt - first) : G;
  const int64_t in = tile - grp * per_group;
  tm = first + in % gsz;
  tn = in / gsz;
}

// First diagonal of the FP64 phase of the fold: diagonals g >= the returned
// value are combined exactly in int64 (the partial sum
// Y = sum_g D_g 2^{beta (S+1-g)} stays below 2^52 by the bound
// |D_g| <= (g-1)(2^beta-1)^2 128 Kt, so the FP64 fold of those steps is
// exact and doing them in integers gives the same bits).
// In integers: seven diagonals of the FP64 form held the FP64 pipe for ~6 us
// per tile with all epilogue threads at it.
__device__ __forceinline__ int oz_exact_from(int S, int beta, int64_t Kt) {
  return ozaki_exact_from(S, beta, Kt);
}

}  // namespace mxm
