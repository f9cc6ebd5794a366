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

// d 2^p as a double (exact), for an int32 d and a normal result.
__device__ __forceinline__ double i32_times_pow2(int d, int p) {
  const uint32_t sign = static_cast<uint32_t>(d) & 0x80000000u;
  const uint32_t mag = static_cast<uint32_t>(d < 0 ? -d : d);  // 2^31 for INT_MIN
  const int lz = __clz(static_cast<int>(mag));
  const uint32_t norm = mag << lz;  // top bit set (mag != 0); lz = 32: shifted out
  const uint32_t hi = sign | (static_cast<uint32_t>(1023 + 31 - lz + p) << 20) |
                      ((norm >> 11) & 0x000FFFFFu);
  const uint32_t lo = norm << 21;
  return __hiloint2double(mag ? static_cast<int>(hi) : 0, mag ? static_cast<int>(lo) : 0);
}

// y 2^p as a double (exact), for |y| < 2^53 and a normal result.
__device__ __forceinline__ double i64_pow2(long long y, int p) {
  const int sg = static_cast<int>(y >> 63);
  const uint64_t mag = static_cast<uint64_t>((y ^ sg) - sg);
  const uint32_t h = static_cast<uint32_t>(mag >> 32), l = static_cast<uint32_t>(mag);
  const bool wide = h != 0;
  const uint32_t top = wide ? h : l, next = wide ? l : 0u;
  const int lz = __clz(static_cast<int>(top));
  const uint32_t n1 = __funnelshift_lc(next, top, lz), n0 = next << (lz & 31);  // normalised
  const uint32_t be = static_cast<uint32_t>(1023 + (wide ? 63 : 31) - lz + p);
  const uint32_t hi = (static_cast<uint32_t>(sg) & 0x80000000u) | (be << 20) |
                      ((n1 >> 11) & 0x000FFFFFu);
  const uint32_t lo = __funnelshift_r(n0, n1, 11);
  return __hiloint2double(top ? static_cast<int>(hi) : 0, top ? static_cast<int>(lo) : 0);
}

// x 2^e: the exponent field moved when x and the result are normal (or x is
// zero), the general form otherwise.
static __device__ __noinline__ double scale_slow(double x, int e) { return ldexp_rn(x, e); }
__device__ __forceinline__ double scale_by(double x, int e) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x));
  const int be = static_cast<int>((hi >> 20) & 0x7FFu);
  const int nb = be + e;
  if (be >= 1 && be <= 2046 && nb >= 1 && nb <= 2046)
    return __hiloint2double(static_cast<int>(hi + (static_cast<uint32_t>(e) << 20)),
                            __double2loint(x));
  return scale_slow(x, e);
}

// y + d 2^sh (sh uniform, a multiple of the digit width, never 31) in int64.
__device__ __forceinline__ long long add_shifted(long long y, int d, int sh) {
  if (sh < 31) return y + static_cast<long long>(d) * (1 << sh);  // one IMAD.WIDE
  return y + static_cast<long long>(static_cast<uint64_t>(static_cast<uint32_t>(d) << (sh - 32)) << 32);
}
__device__ __forceinline__ long long add_shifted(long long y, long long d, int sh) {
  return y + static_cast<long long>(static_cast<uint64_t>(d) << sh);
}
__device__ __forceinline__ double sum_pow2(int d, int p) { return i32_times_pow2(d, p); }
__device__ __forceinline__ double sum_pow2(long long d, int p) { return i64_pow2(d, p); }

}  // namespace mxm
