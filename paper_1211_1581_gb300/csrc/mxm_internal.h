// mxm_internal.h -- declarations shared by the translation units of
// libmxm.so (not part of the public C ABI in include/mxm.h).
#pragma once
#include <cstddef>
#include <atomic>
#include <cstdint>

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <utility>

namespace mxm {

// A named NVTX range around one ABI call (scope-bound), so that a profiler's
// timeline shows which call launched which kernels.  Without a profiler
// attached NVTX calls return at once.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

// Bits of the sticky device status word (OR-ed by kernels).
constexpr int kStatusNonFinite = 1;
constexpr int kStatusTimeout = 2;
constexpr int kStatusWorkspace = 4;
constexpr int kStatusBounds = 8;
constexpr int kStatusBreakdown = 16;

// Every bounded wait inside a kernel gives up after this long (the barriers of
// cg_grid.cu, where the others may be at work on long rows, later: cg_rows.h).
constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s

// Split-k for products with fewer C tiles than SMs: the k-blocks of every
// tile are cut into `splits` contiguous ranges, each computed by its own
// CTA into a partial tile; a second kernel adds the partials in split order
// (a fixed order: the result does not depend on timing).  The number of
// work units aimed at is a constant (two per SM of a 152-SM GB300), not the
// device's SM count, so that a product's rounding does not depend on the
// device it runs on; every range keeps at least `min_blocks` k-blocks.
constexpr int64_t kSplitKUnits = 304;

inline int64_t splitk_count(int64_t tiles, int64_t Kt, int64_t min_blocks) {
  if (tiles <= 0 || tiles >= kSplitKUnits / 2) return 1;
  int64_t s = kSplitKUnits / tiles;
  const int64_t cap = Kt / min_blocks;
  if (s > cap) s = cap;
  return s > 1 ? s : 1;
}

// ---------------------------------------------------------------- Ozaki
// Operand tiles of the slice GEMM: 128 rows x 128 bf16, 32 KiB, stored
// pre-swizzled so that one bulk copy moves a tile into shared memory in the
// layout tcgen05.mma reads: two 128-byte-swizzle atoms along k (k 0..63 and
// 64..127, 16 KiB each), each with rows of 128 bytes in which the 16-byte
// chunk c of row r sits at chunk position c ^ (r % 8).  (Bulk copies of
// 32 KiB stream about twice as fast per SM as copies of 16 KiB.)
constexpr int kOzTileRows = 128;
constexpr int kOzTileK = 128;
constexpr int kOzAtomK = 64;
constexpr int kOzAtomBytes = kOzTileRows * kOzAtomK * 2;
constexpr int kOzTileBytes = kOzTileRows * kOzTileK * 2;
constexpr int kOzChunksPerRow = kOzTileK / 8;

// Byte offset of 16-byte chunk c (k = 8c .. 8c+7) of row r inside a tile.
__host__ __device__ inline int oz_chunk_offset(int r, int c) {
  return (c >> 3) * kOzAtomBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4);
}
constexpr int kOzMaxSlices = 12;

// B tiles for the CTA-pair product (cta_group::2, M = 256): the tile's rows
// (columns of B) in two halves of 64, each half contiguous (16 KiB: its two
// atoms along k of 64 rows x 128 bytes, 8 KiB each), so that each CTA of a
// pair fetches its half with one bulk copy.  Same swizzle: chunk c of row r
// at chunk position c ^ (r % 8).
__host__ __device__ inline int oz_chunk_offset_halves(int r, int c) {
  return (r >> 6) * (kOzTileBytes / 2) + (c >> 3) * (kOzAtomBytes / 2) + (r & 63) * 128 +
         (((c & 7) ^ (r & 7)) << 4);
}

// The 4-bit-digit engine: digits |d| <= 15 carried in FP8 E4M3 (every
// integer up to 16 is exact there) through tcgen05 kind::f8f6f4.  A tile is
// 128 rows x 128 k of one byte: a single 128-byte-swizzle atom of 16 KiB, the
// 16-byte chunk c (k = 16c .. 16c+15) of row r at chunk position c ^ (r % 8).
constexpr int kOzTileBytesE4m3 = kOzTileRows * kOzTileK;
constexpr int kOzMaxSlicesE4m3 = 16;
constexpr int kOzMaxSlicesRn8 = 7;
__host__ __device__ inline int oz_chunk_offset_e4m3(int r, int c) {
  return r * 128 + ((c ^ (r & 7)) << 4);
}

struct OzakiDims {
  int64_t m, k, n;
  int64_t Mt, Nt, Kt;  // tiles of 128 rows of A, 128 columns of B, 128 of k
  int S, beta;
  int64_t splits;      // k ranges per C tile (1: no split-k)
  int fp8;             // 1: digits carried in E4M3 (beta = 4), 0: in bf16
  int rn;              // 1: balanced 8-bit digits, the value rounded once to
                       //    nearest (beta = 8, scale exponent + 1, |d| <= 128)
  int pair;            // 1: the slice GEMM runs on CTA pairs (cta_group::2) and
                       //    the B digit tiles are written in the halves layout
  int raster;          // tile-rows (pair-rows on CTA pairs) per group of the
                       //    persistent walk over C tiles
  int kb_alt;          // 1: alternate the k-block direction from one diagonal
                       //    (pair) to the next
  int kara;            // 1: difference products on 256 x 256 C tiles (ozaki_kara.cu),
                       //    2: on 256 x 128 tiles (little k); the operands have
                       //    kara_planes(S) digit planes
  int chain;           // 1: the launches of the product follow one another on one
                       //    stream (launch_chained)
};

// Default walk: groups of 8 tile-rows (4 pair-rows on CTA pairs); the
// emulated modes alternate the k-block direction between diagonal pairs.
constexpr int kDefaultRaster = 8;
constexpr int kPairRaster = 4;

inline OzakiDims ozaki_dims(int64_t m, int64_t k, int64_t n, int S, int beta, bool rn = false) {
  OzakiDims d;
  d.m = m; d.k = k; d.n = n;
  d.Mt = (m + kOzTileRows - 1) / kOzTileRows;
  d.Nt = (n + kOzTileRows - 1) / kOzTileRows;
  d.Kt = (k + kOzTileK - 1) / kOzTileK;
  d.S = S; d.beta = beta;
  d.splits = 1;
  d.fp8 = 0;
  d.rn = rn ? 1 : 0;
  d.pair = d.Mt >= 2 ? 1 : 0;
  d.raster = kDefaultRaster;
  d.kb_alt = 0;
  d.kara = 0;
  d.chain = 0;
  return d;
}

// Largest digit magnitude of a split.
inline int ozaki_dmax(const OzakiDims& d) { return d.rn ? 128 : (1 << d.beta) - 1; }

// The 4-bit-digit E4M3 engine (paired kernel only: no split-k).
inline OzakiDims ozaki_dims_fp8(int64_t m, int64_t k, int64_t n, int S) {
  OzakiDims d = ozaki_dims(m, k, n, S, 4);
  d.fp8 = 1;
  d.pair = 0;
  return d;
}

inline size_t ozaki_tile_bytes(const OzakiDims& d) {
  return d.fp8 ? kOzTileBytesE4m3 : kOzTileBytes;
}

// The same with split-k where the product has fewer C tiles than SMs (each
// k range at least 4 k-blocks of 128): the per-range digit-pair sums D_g
// are exact integers, added exactly, so the result is bit-identical to the
// unsplit product.
inline OzakiDims ozaki_dims_splitk(int64_t m, int64_t k, int64_t n, int S, int beta,
                                   bool rn = false) {
  OzakiDims d = ozaki_dims(m, k, n, S, beta, rn);
  d.splits = splitk_count(d.Mt * d.Nt, d.Kt, 4);
  if (d.splits > 1) d.pair = 0;
  return d;
}

// Whether the B digit tiles are written in the halves layout above, and
// whether the paired slice GEMM runs on CTA pairs (cta_group::2, 256-row C
// tiles): bf16 digits without split-k, chosen where the dims are made (two
// or more tile-rows of A; products that share B planes share the choice,
// a single tile-row then leaving the second CTA of its pairs idle).
inline bool ozaki_b_halves(const OzakiDims& d) { return d.pair != 0 && !d.fp8 && d.kara != 1; }
inline bool ozaki_cta2(const OzakiDims& d) {
  return ozaki_b_halves(d) && d.splits <= 1 && d.Mt >= 1;
}

// Workspace layout of one emulated product (offsets in bytes, 1 KiB aligned).
struct OzakiLayout {
  size_t rowbits, colbits, aslices, bslices, sums, total;
};

__host__ __device__ inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Whether the per-diagonal integer sums of a tile with Kt k-blocks fit in
// int32, the condition of the paired slice GEMM without spills: every digit
// product is at most (2^beta - 1)^2 and a diagonal has at most S of them
// per k.
__host__ __device__ inline bool ozaki_narrow(int S, int beta, int64_t Kt) {
  const double dmax = static_cast<double>((1 << beta) - 1);
  return static_cast<double>(S) * dmax * dmax * kOzTileK * static_cast<double>(Kt) <
         2147483647.0;
}

// The same for the dims of a product (the digit bound of its split).
inline bool ozaki_narrow(const OzakiDims& d) {
  const double dmax = static_cast<double>(d.rn ? 128 : (1 << d.beta) - 1);
  return static_cast<double>(d.S) * dmax * dmax * kOzTileK * static_cast<double>(d.Kt) <
         2147483647.0;
}

// CTAs of the paired slice GEMM that keep a spill area (the grid is capped
// there when spills are on).
constexpr int64_t kOzSpillCtas = 256;

// Bytes of the running sums of a product (per C tile 128 x 128 x 8 bytes),
// or under split-k the partial sums D_g of every k range.
inline size_t ozaki_sums_bytes(const OzakiDims& d) {
  const size_t tile8 = (size_t)kOzTileRows * kOzTileRows * 8;
  return d.splits > 1 ? (size_t)d.splits * d.Mt * d.Nt * d.S * tile8
                      : (size_t)d.Mt * d.Nt * tile8;
}

// Spill area of the paired slice GEMM when a diagonal's integer sum can
// outgrow int32 over all of k (long k, 8-bit digits): per CTA the int64
// partial sums of the two diagonals in work, 2 x 128 x 128 x 8 bytes.
inline size_t ozaki_spill_bytes(const OzakiDims& d) {
  if (d.fp8 || d.splits > 1 || ozaki_narrow(d)) return 0;
  const int64_t ctas = d.Mt * d.Nt < kOzSpillCtas ? d.Mt * d.Nt : kOzSpillCtas;
  return (size_t)ctas * 2 * kOzTileRows * kOzTileRows * 8;
}

// Largest number of K=16 MMAs whose integer products can be summed in an
// FP32 accumulator without rounding: every product is at most (2^beta-1)^2
// in magnitude and 16 of them enter per MMA, so the running sum stays within
// 2^24 (all integers up to 2^24 are exact in FP32).
inline int ozaki_window_mmas(int beta, bool rn = false) {
  const long long dmax = rn ? 128 : (1ll << beta) - 1;
  const long long per_mma = dmax * dmax * 16;
  return static_cast<int>((1ll << 24) / per_mma);
}

// The same bound in whole k-blocks (kOzTileK / 16 MMAs each), as the kernel
// counts.
inline int ozaki_window_stages(int beta, bool rn = false) {
  return ozaki_window_mmas(beta, rn) / (kOzTileK / 16);
}

// ---------------------------------------------------------------- difference products
// (ozaki_kara.cu; the identity is stated there.)  Digit planes of an operand:
// the S digits, then one difference plane for every pair s < t with
// s + t <= S + 1 except (1, S), ordered by s + t, then s.
constexpr int kKaraMaxSlices = 9;
__host__ __device__ inline int kara_pairs(int S) {
  int n = -1;
  for (int g = 3; g <= S + 1; ++g) n += (g - 1) / 2;
  return n > 0 ? n : 0;
}
__host__ __device__ inline int kara_planes(int S) { return S + kara_pairs(S); }
inline int kara_pair_plane(int S, int s, int t) {
  int idx = S;
  for (int g = 3; g < s + t; ++g) idx += (g - 1) / 2;
  idx += s - 1;
  if (s + t == S + 1) --idx;  // (1, S) has no plane
  return idx;
}

// Exact FP32 windows (k-blocks) of the difference products: truncated digits
// of one value have one sign, so their differences keep the digit bound;
// balanced digits differ by at most 256.
inline int kara_window_stages(const OzakiDims& d) {
  return d.rn ? static_cast<int>((1ll << 24) / (256ll * 256 * 16)) / (kOzTileK / 16)
              : ozaki_window_stages(d.beta, false);
}

// Most products in one segment: N_{S+1} (the pair (1, S) counts twice).
inline int kara_max_segment(int S) { return S / 2 + 1; }

// 256 x 256 C tiles of the CTA pairs; the pairs of a 152-SM GPU (a constant,
// so that the workspace is host arithmetic); the scratch: S slots per tile
// and CTA of the pair, and those of the tiles cut into units (fewer than the
// pairs, or all where k is cut for the sums' sake; 2 S - 2 slots per tile and
// k range; the cut stays within them).
constexpr int64_t kKaraPairs = 76;
constexpr size_t kKaraSlotBytes = (size_t)kOzTileRows * 256 * 4;
inline int64_t kara_tiles(const OzakiDims& d) { return (d.Mt + 1) / 2 * ((d.Nt + 1) / 2); }
// The k ranges that keep every sum of a range in int32 (1 unless k is long for
// the digits: S = 6 of 8 bits beyond k = 5,504).  Measured against the digit
// products one by one with spills (8-bit digits, S = 6): 2048 x 8192 x 2048
// 1670 -> 1176 us, 4096 x 8192 x 4096 5515 -> 3723 us.
inline int kara_min_ranges(const OzakiDims& d) {
  if (ozaki_narrow(d)) return 1;
  const double dmax = static_cast<double>(ozaki_dmax(d));
  const int64_t most =
      static_cast<int64_t>(2147483647.0 / ((d.S + 1) * dmax * dmax * kOzTileK));
  return most < 1 ? 0 : static_cast<int>((d.Kt + most - 1) / most);
}
// The most ranges a cut takes: at least four k-blocks each otherwise.
inline int kara_max_ranges(const OzakiDims& d) {
  const int64_t least = kara_min_ranges(d), most = least > d.Kt / 4 ? least : d.Kt / 4;
  return static_cast<int>(most < least + 15 ? most : least + 15);
}
inline size_t kara_cut_slots(const OzakiDims& d) {
  const int64_t t = kara_tiles(d), r = kara_min_ranges(d);
  const int64_t cut = t < kKaraPairs || r > 1 ? t : kKaraPairs;
  const size_t one = (size_t)cut * (2 * d.S - 2), least = one * r;
  const size_t most = one * kara_max_ranges(d), cap = 3 * (size_t)kKaraPairs;
  return most <= cap ? most : (least > cap ? least : cap);
}
inline size_t kara_scratch_bytes(const OzakiDims& d) {
  if (d.kara == 2) {  // per CTA S slots of a 128 x 128 tile
    const int64_t t = (d.Mt + 1) / 2 * d.Nt;
    return kKaraSlotBytes * (size_t)(t < kKaraPairs ? t : kKaraPairs) * d.S;
  }
  const size_t whole = kara_min_ranges(d) > 1 ? 0 : (size_t)kara_tiles(d) * d.S;
  return 2 * kKaraSlotBytes * (whole + kara_cut_slots(d));
}

// The first diagonal of the FP64 phase of the fold (oz_exact_from).
__host__ __device__ inline int ozaki_exact_from(int S, int beta, int64_t Kt) {
  const uint64_t dmax = (1u << beta) - 1;
  const uint64_t one = dmax * dmax * kOzTileK * static_cast<uint64_t>(Kt);  // < 2^48
  int gx = S + 1;
  uint64_t y = 0;
  for (int g = S + 1; g >= 2; --g) {
    const int sh = beta * (S + 1 - g);
    const uint64_t d = static_cast<uint64_t>(g - 1) * one;
    if (sh >= 52 || (d >> (52 - sh)) != 0) break;  // this diagonal alone reaches 2^52
    y += d << sh;
    if (y >> 52) break;
    gx = g;
  }
  return gx;
}

// Which products can take the difference products.
inline bool kara_fits(const OzakiDims& d) {
  return !d.fp8 && d.S >= 3 && d.S <= kKaraMaxSlices && d.beta * d.S <= 64 && d.Kt > 0 &&
         kara_min_ranges(d) >= 1 && kara_min_ranges(d) <= 16 &&
         d.Mt >= 1 && d.Nt >= 1 && kara_tiles(d) < (1 << 24);
}

inline OzakiLayout ozaki_layout(const OzakiDims& d) {
  OzakiLayout L;
  size_t off = 0;
  L.rowbits = off; off = align_up(off + sizeof(uint64_t) * (size_t)(d.m > 0 ? d.m : 1), 1024);
  L.colbits = off; off = align_up(off + sizeof(uint64_t) * (size_t)(d.n > 0 ? d.n : 1), 1024);
  const size_t planes = d.kara ? kara_planes(d.S) : d.S;
  L.aslices = off; off = align_up(off + planes * d.Mt * d.Kt * ozaki_tile_bytes(d), 1024);
  L.bslices = off; off = align_up(off + planes * d.Nt * d.Kt * ozaki_tile_bytes(d), 1024);
  if (d.kara) {  // the segment sums of the difference-product kernel
    L.sums = off;
    L.total = align_up(off + kara_scratch_bytes(d), 1024);
    return L;
  }
  // running sums of the recombination between diagonal pairs: per C tile
  // 128 x 128 x 8 bytes, column-major inside the tile (so that a warp, which
  // owns 32 consecutive rows, touches 256 contiguous bytes per column).
  // Under split-k the region holds instead the int64 partial sums D_g of
  // every k range: [splits][Mt x Nt tiles][S diagonals] x 128 x 128,
  // column-major inside the tile.  The spill area (if any) follows the sums.
  L.sums = off; off = align_up(off + ozaki_sums_bytes(d), 1024);
  off = align_up(off + ozaki_spill_bytes(d), 1024);
  L.total = off;
  return L;
}


constexpr int kKaraShortSlices = 7;
// The choice: the workspace (digit and difference planes, segment slots) up
// to kKaraMaxBytes (6.8 GB at 8192^3, 27 GB at 16384^3); not for a part of a
// wave with little k, where the planes and slots cost more than the products
// save (measured at 512 x 512 x 4096, S = 7: 154 us against 148); and with a
// single tile-row or tile-column, where half of a 256 x 256 tile is empty,
// only as long as the product is small enough to be bound by latency (155 x
// 305 x 98, S = 7: 3x; 64 x 8192 x 8192, S = 6: 956 us against 906).  Against the
// one-by-one products as they are now, over 294 products that take the difference
// products: 1.59 times as fast in the geometric mean, 21 of them slower, most
// one tile-row beside many tile-columns with two k-blocks (128 x 200 x 16384, S =
// 8: 154 us against 127).
constexpr size_t kKaraMaxBytes = (size_t)32 << 30;
// Little k: 256 x 128 tiles, where the epilogue sets the pace and there are
// tiles for most CTA pairs.  Measured against 256 x 256 tiles (S = 7): up to
// three k-blocks (4096 x 128 x 4096 255 us against 384, 16384 x 256 x 16384 4.5
// ms against 5.6, 2048 x 256 x 2048 121 against 134), four with many tiles (8192 x
// 512 x 8192 1780 against 1859, but 2048 x 512 x 2048 175 against 169), up to
// eight where all tiles are one wave (1024 x 512 x 2048 109 against 126).
inline bool kara_short(const OzakiDims& d) {
  if (!kara_fits(d) || !ozaki_narrow(d) || d.S > kKaraShortSlices || d.Mt < 2) return false;
  const int64_t tiles = (d.Mt + 1) / 2 * d.Nt;
  if (tiles < 40) return false;
  return d.Kt <= 3 || (d.Kt <= 4 && tiles >= 512) || (d.Kt <= 8 && tiles <= kKaraPairs);
}
// One k-block of one tile-row or tile-column: one by one, a lone CTA takes the
// diagonals of a tile in turn; here the segments are shared out over the SMs
// (64^3, S = 7: 35 us against 74; 4096 x 64 x 64, 16 tiles, 52 against 81; with
// 64 tiles there is a CTA for each: 16384 x 64 x 64 74 against 75).  Apart from
// kara_chosen because a caller is not asked for its workspace (workspace_told).
inline bool kara_one_block(const OzakiDims& d) {
  return kara_fits(d) && d.Kt == 1 && (d.Mt == 1 || d.Nt == 1) && kara_tiles(d) <= 16;
}
inline bool kara_chosen(const OzakiDims& d) {
  if (!kara_fits(d)) return false;
  const bool is_short = kara_short(d);
  if (!is_short && d.Kt <= 4 && kara_tiles(d) > 16 && kara_tiles(d) < 48) return false;
  if (!is_short && (d.Mt == 1 || d.Nt == 1) && (d.Kt < 2 || kara_tiles(d) * d.Kt > 256)) return false;
  OzakiDims w = d;
  w.kara = is_short ? 2 : 1;
  return ozaki_layout(w).total <= kKaraMaxBytes;
}

// The plan of ozaki_dims_splitk when its workspace fits `cap` bytes, else
// the same product without split-k (the split-k partials are exact integers
// added exactly, so both plans give the same bits).  The caller checks
// whether the returned plan fits.
inline OzakiDims ozaki_dims_capped(int64_t m, int64_t k, int64_t n, int S, int beta,
                                   size_t cap) {
  OzakiDims d = ozaki_dims_splitk(m, k, n, S, beta);
  if (d.splits > 1 && ozaki_layout(d).total > cap) d = ozaki_dims(m, k, n, S, beta);
  return d;
}

cudaError_t launch_ozaki_scale(const double* A, const double* B, const OzakiDims& d,
                               uint64_t* rowbits, uint64_t* colbits, int* status,
                               cudaStream_t s);
// Splits A and B into digit planes.  For bf16 digits with k up to 24576 the
// row maxima of A are found here too (one pass over A: launch_ozaki_scale then
// does B only), so rowbits is written and status takes a non-finite A.
cudaError_t launch_ozaki_split(const double* A, const double* B, const OzakiDims& d,
                               uint64_t* rowbits, const uint64_t* colbits,
                               uint8_t* aslices, uint8_t* bslices, int* status, cudaStream_t s);
cudaError_t launch_ozaki_gemm(const uint8_t* aslices, const uint8_t* bslices,
                              const uint64_t* rowbits, const uint64_t* colbits, double* C,
                              const OzakiDims& d, uint64_t* sums, int* status, cudaStream_t s);
// The same by difference products (d.kara; scratch: kara_scratch_bytes(d)).
cudaError_t launch_ozaki_kara(const uint8_t* aslices, const uint8_t* bslices,
                              const uint64_t* rowbits, const uint64_t* colbits, double* C,
                              const OzakiDims& d, uint8_t* scratch, int* status, cudaStream_t s);

// ---------------------------------------------------------------- FP64
constexpr int kF64BM = 128, kF64BN = 128, kF64BK = 16;
constexpr int kF64TileBytes = kF64BM * kF64BK * 8;  // 16 KiB (BM == BN)

struct F64Dims {
  int64_t m, k, n, Mt, Nt, Kt;
  int64_t splits;  // k ranges per 128 x 128 tile the workspace has room for
  int64_t ranges;  // where a worker's share may end along k: 0 after any step,
                   // s at the s-ths of k (1: not inside a piece)
};

inline F64Dims f64_dims(int64_t m, int64_t k, int64_t n) {
  F64Dims d;
  d.m = m; d.k = k; d.n = n;
  d.Mt = (m + kF64BM - 1) / kF64BM;
  d.Nt = (n + kF64BN - 1) / kF64BN;
  d.Kt = (k + kF64BK - 1) / kF64BK;
  d.splits = splitk_count(d.Mt * d.Nt, d.Kt, 8);
  // little k: pieces are not cut (a piece is at most 8 steps, 34 us)
  d.ranges = k < 32 ? 1 : 0;
  return d;
}

// The workers of the native product (two warps on each of the 608 SM
// sub-partitions of a 152-SM GPU, each with at least one step of 8 DMMAs) and
// the two 32 x 32 slots (and its place in a table of the shares' starts) each
// needs when shares cut pieces.
constexpr int64_t kF64Piece = 32;
constexpr size_t kF64WorkerBytes = 2 * kF64Piece * kF64Piece * sizeof(double) + 16;
inline int64_t f64_workers(const F64Dims& d) {
  const int64_t steps = (d.m + 15) / 16 * ((d.n + 7) / 8) * ((d.k + 3) / 4) / 8;
  return steps < 1 ? 1 : (steps < 1216 ? steps : 1216);
}

// Workspace of a native product: the workers' slots, 20 MB at most, and what the
// library allocates for it.
inline size_t f64_workspace(const F64Dims& d) {
  return d.ranges == 1 ? 0 : (size_t)(f64_workers(d) + 1) * kF64WorkerBytes;
}
// The size that an earlier form of the product needed, zero-padded 128 x 16 tile
// copies of A and B and the partial tiles of the k ranges: buffers of it are
// kept by callers.  A product runs in the smaller of the two, and callers are
// told the larger.
inline size_t f64_workspace_kept(const F64Dims& d) {
  const size_t packs = align_up((size_t)(d.Mt + d.Nt) * d.Kt * kF64TileBytes, 1024);
  const size_t partials =
      d.splits > 1 ? (size_t)d.splits * d.Mt * d.Nt * kF64BM * kF64BN * sizeof(double) : 0;
  return align_up(packs + partials, 1024);
}
inline size_t f64_workspace_least(const F64Dims& d) {
  const size_t slots = f64_workspace(d), kept = f64_workspace_kept(d);
  return slots < kept ? slots : kept;
}
inline size_t f64_workspace_told(const F64Dims& d) {
  const size_t slots = f64_workspace(d), kept = f64_workspace_kept(d);
  return slots > kept ? slots : kept;
}

// C = A.B with ws_bytes of workspace (fewer slots: fewer workers).
cudaError_t launch_f64_gemm(const double* A, const double* B, double* C, const F64Dims& d,
                            uint8_t* ws, size_t ws_bytes, int* status, cudaStream_t s);

cudaError_t launch_zero_fill(double* C, int64_t count, cudaStream_t s);

// ---------------------------------------------------------------- grouped
// Device plan of a grouped call, written by grouped_plan_kernel at the start
// of the caller's workspace: a header, one record per problem (with prefix
// sums of every per-problem count), then the data regions.
struct GroupedProblem {
  const double* A;
  const double* B;
  double* C;
  int64_t m, k, n;
  int64_t Mt, Nt, Kt;      // 128-row tiles of A, 128-column tiles of B, k-blocks
  int64_t tile_begin;      // first C tile (prefix of Mt*Nt)
  int64_t atile_begin;     // first A operand tile (prefix of Mt*Kt)
  int64_t btile_begin;     // first B operand tile (prefix of Nt*Kt)
  int64_t row_begin;       // first row maximum (prefix of m)
  int64_t col_begin;       // first column maximum (prefix of n)
  int64_t trow_begin;      // first tile-row of A (prefix of Mt)
  int64_t tcol_begin;      // first tile-column of B (prefix of Nt)
  int64_t ltile_begin;     // emulated: first C tile among the long-k problems
  int64_t stile_begin;     // emulated: first C tile among the short-k problems
};

struct GroupedHeader {
  int64_t valid;           // 0: workspace too small, every later kernel does nothing
  int64_t count;           // problems
  int64_t tiles, atiles, btiles, rows, cols, trows, tcols, ltiles, stiles, max_kt;
  int64_t off_rowbits, off_colbits, off_a, off_b, total;  // byte offsets in the workspace
  int64_t cursor;          // next work unit of a dynamically scheduled kernel (zeroed by
                           // the plan kernel on every call)
  int64_t off_sums, off_spill;  // emulated: running sums of every C tile, spill areas
  int64_t cursor_max;      // next unit of the emulated maxima pass (zeroed like cursor)
  int64_t off_owner;       // emulated: the problem (int32) owning each A tile, B tile,
                           // short-k C tile, long-k C tile, A tile-row and B
                           // tile-column, in that order
};

constexpr size_t kGroupedRecordsOff = 256;
static_assert(sizeof(GroupedHeader) <= kGroupedRecordsOff, "the header precedes the records");

__host__ __device__ inline size_t grouped_data_begin(int64_t count) {
  return align_up(kGroupedRecordsOff + sizeof(GroupedProblem) * static_cast<size_t>(count), 1024);
}

// Byte offsets of the data regions from the totals (same on host and device).
__host__ __device__ inline void grouped_offsets(GroupedHeader& h, int planes, size_t tile_bytes,
                                                bool bits) {
  size_t off = grouped_data_begin(h.count);
  h.off_rowbits = off;
  if (bits) off = align_up(off + 8 * static_cast<size_t>(h.rows > 0 ? h.rows : 1), 1024);
  h.off_colbits = off;
  if (bits) off = align_up(off + 8 * static_cast<size_t>(h.cols > 0 ? h.cols : 1), 1024);
  h.off_a = off;
  off = align_up(off + static_cast<size_t>(planes) * h.atiles * tile_bytes, 1024);
  h.off_b = off;
  off = align_up(off + static_cast<size_t>(planes) * h.btiles * tile_bytes, 1024);
  // emulated: the running sums of the diagonal-pair slice GEMM (128 x 128 x 8
  // bytes per C tile of the long-k problems) and the int64 spill areas of its
  // CTAs (long k)
  h.off_sums = off;
  if (bits) off = align_up(off + static_cast<size_t>(h.ltiles) * kOzTileRows * kOzTileRows * 8, 1024);
  h.off_spill = off;
  if (bits) off = align_up(off + static_cast<size_t>(kOzSpillCtas) * 2 * kOzTileRows * kOzTileRows * 8,
                           1024);
  h.off_owner = off;
  if (bits)
    off = align_up(off + 4 * static_cast<size_t>(h.atiles + h.btiles + h.stiles + h.ltiles +
                                                 h.trows + h.tcols + 1),
                   1024);
  h.total = off;
}

// Index of the problem owning item t of the prefix field `begin`: the last
// record whose begin is <= t (problems with no items share their begin with
// the next one and are skipped by "last").
template <typename Rec>
__device__ __forceinline__ int64_t grouped_find(const Rec* recs, int64_t count, int64_t t,
                                                int64_t Rec::*begin) {
  int64_t lo = 0, hi = count - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (recs[mid].*begin <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Problems of a grouped emulated call with at most this many k-blocks run on
// the one-diagonal slice GEMM (running sums in tensor memory), the others on
// the diagonal-pair GEMM.
// Measured on 2000 problems of dims log-uniform in [16, 1024] (k <= 8 blocks):
// all on the one-diagonal kernel is fastest (11.0 ms at S = 8 against 14.4 ms
// all on the pair kernel), so the default takes every problem up to 8 blocks.
constexpr int kGroupedShortKt = 8;
// short_kt: the plan's boundary (k-blocks) between the short-k problems (the
// one-diagonal kernel) and the long-k ones (the diagonal-pair kernel).
cudaError_t launch_ozaki_grouped(uint8_t* ws, int S, int beta, int64_t short_kt, int* status,
                                 cudaStream_t s, bool rn = false);
// Native grouped products: work units of 32 x 32 C elements (one warp each,
// operands loaded straight from the caller's arrays, k in steps of 4).
constexpr int kF64GroupedTile = 32;
constexpr int kF64GroupedK = 4;
cudaError_t launch_f64_grouped(uint8_t* ws, int* status, cudaStream_t s);
int sm_count();

// A property of one kernel (or one launch shape) on each device, asked for
// once: that its dynamic shared memory limit is raised, how many clusters the
// device holds.  Kept at the launch site in a static of this type; two
// threads that come first together both ask, with the same answer; a failed
// question is asked again.  The limit is raised to the most that the site
// uses, so calls of different sizes do not lower it under each other.  The
// calls cost host time on every launch: a lone transform of 256 points, bound
// by the host, 19.4 -> 18.3 us, of 8192 23.6 -> 22.7.
class PerDevice {
 public:
  template <typename Make>  // Make: cudaError_t(int* value), value >= 0
  cudaError_t get(int* value, Make&& make) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool kept = dev >= 0 && dev < kDevices;
    int v = kept ? known_[dev].load(std::memory_order_acquire) - 1 : -1;
    if (v < 0) {
      if ((e = make(&v)) != cudaSuccess) return e;
      if (kept) known_[dev].store(v + 1, std::memory_order_release);
    }
    *value = v;
    return cudaSuccess;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> known_[kDevices] = {};
};

// Launch a kernel that begins with follow_grid() or ends with it (ptx.cuh) while
// the kernel before it on the stream still runs (chain; programmatic dependent
// launch): its blocks take the SMs that the earlier grid no longer fills, set
// up and wait there.  Every thread of such a kernel waits before its first
// access to what an earlier kernel of the call wrote, and every thread of
// every such kernel waits at some point, so that its end implies the end of
// all the kernels before it.  Small calls are mostly the gaps between their
// launches: 256^3 emulated (S = 7, five kernels) 42 -> 30 us, 256^3 native
// 51.8 -> 47.8, 1000 x 1777 x 1300 emulated 164 -> 153, a transform of 2^16 points
// 20.5 -> 18.5, of 2^20 163.9 -> 157.8.
template <typename... P, typename... Q>
cudaError_t launch_chained(bool chain, void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                           cudaStream_t s, Q&&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Q>(args)...);
}

// Raise a kernel's dynamic shared memory limit on the current device.
template <typename Kernel>
cudaError_t allow_smem(PerDevice& site, Kernel kern, size_t bytes) {
  int done = 0;
  return site.get(&done, [&](int* v) {
    *v = 1;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(bytes));
  });
}

// Whether the fold of a split-k product of m rows, `blocks` blocks of it, is
// launched beside the slice GEMM.  The GEMM's CTAs leave no registers for a fold
// block, so blocks launched early all settle on the first SMs that are free; with
// few rows every lane of their loads is a sector of its own, and those SMs are
// long at it.  S = 7, beside against after: 1 x 4096 x 4096 402 us against 281, 4
// rows 299 against 275, 8 rows 282 against 274, 16 rows 277 against 276; 1 x 65536
// x 1 (one block) 157 against 160.
inline bool splitk_fold_chained(int64_t m, int64_t blocks) { return m >= 16 || blocks <= 8; }

// ---------------------------------------------------------------- FFT
constexpr int kFftThreads = 256;

// log2 of the columns per CTA of a pass over `cols` transforms of 2^bits points (a
// power of two, at most 8, at most 96 KiB of shared memory): the most for which
// the last wave of CTAs over the SMs is at least 0.9 full on average over the
// waves, else the count with the fullest waves; of equally full ones the fewest
// columns that leave every thread of a CTA a butterfly of four points.  Fewer
// CTAs than SMs have too few warps to hide latency: 2^19 points with 128 CTAs of
// four columns in the first pass 121 us, 512 of one 101; 2^18 with 128 of four in
// both 59.1, 256 of two 57.0; but 2^17 with less than 1024 points a CTA 38.6
// instead of 36.6.
inline int fft_column_bits(int bits, int64_t cols, int64_t sms) {
  int best = 0;
  double best_fill = 0.0;
  for (int cb = 3; cb >= 0; --cb) {
    const int64_t C = int64_t{1} << cb, L = int64_t{1} << bits;
    if (cols < C || (C * L + L) * 16 > 96 * 1024) continue;
    const int64_t blocks = cols / C;
    const double fill = static_cast<double>(blocks) / static_cast<double>((blocks + sms - 1) / sms * sms);
    if (fill >= 0.9) return cb;
    if (fill > best_fill || (fill == best_fill && C * L >= 4 * kFftThreads)) {
      best_fill = fill;
      best = cb;
    }
  }
  return best;
}

// Comparison modes (not FP64-accurate).
cudaError_t launch_bf16_gemm(const double* A, const double* B, double* C, const OzakiDims& d,
                             uint8_t* aplane, uint8_t* bplane, int* status, cudaStream_t s);
cudaError_t launch_f32_gemm(const double* A, const double* B, double* C, int64_t m, int64_t k,
                            int64_t n, cudaStream_t s);

}  // namespace mxm
