// ozaki_kara.cu -- steps 3-4 of the Ozaki product (see ozaki.cu) with fewer
// digit products: Karatsuba's identity (Karatsuba and Ofman, 1962) on the
// digit planes.
//
// For two slices s < t of one operand pair
//   A_s B_t + A_t B_s = A_s B_s + A_t B_t + (A_s - A_t)(B_t - B_s),
// so with P_s = A_s B_s and the difference products M_st = (A_s - A_t)(B_t - B_s)
//   D_g = sum_{s < g} P_s + sum_{s + t = g, s < t} M_st
// (the middle square P_{g/2} is among the P_s).  The S - 1 squares P_1 ..
// P_{S-1} serve every diagonal; the pair (1, S) is taken directly (A_1 B_S and
// A_S B_1: a difference product would need P_S as well, which nothing else
// reads), D_{S+1} then leaving out P_1.  S = 7: 19 products instead of 28
// (6: 15 of 21; 8: 24 of 36).  All sums are exact integers, so D_g and the
// result have the same bits as with the products taken one by one.  The
// truncated digits of one value all carry its sign, so |a_s - a_t| is at most
// the digit bound 2^beta - 1: a difference plane is as exact in bf16, and its
// products fill an exact FP32 window as slowly, as the digits themselves.
// Balanced digits (|d| <= 128) differ by at most 256 (exact in bf16; windows
// of 16 MMAs for the M_st).  The split writes the difference planes after the
// digit planes.
//
// Kernel.  Every product has its own A and B plane, so no operand tile is
// shared between two products as in the diagonal-pair kernel; C tiles of
// 256 x 256 on CTA pairs (cta_group::2, M = N = 256: each CTA holds 128 rows
// of A and 128 columns of B) halve the operand bytes per MMA instead: 64 KiB
// per SM and k-block of 8 MMAs (66 ns each).  Tensor memory holds two windows
// of 256 columns.  A tile runs through a list of segments, each the sum of a
// few products: first the squares P_s, then the diagonals' own parts
// N_g = sum M_st (and the pair (1, S)).  Sixteen epilogue warps add the windows
// of a segment into 64 int32 registers per thread (modulo 2^32: only the D_g
// have to fit).  The squares are summed up, T_g = P_1 + .. + P_{g-1}, and each
// T_g is left in its slot of the scratch; a diagonal's part then starts from
// T_g instead of 0 (the slot is read while its first window is computed) and
// leaves D_g.  The recombination is a kernel of its own (oz_kara_fold_kernel,
// HBM-bound): inside this one it held up the MMAs, the two windows in flight
// covering only 8 us of it.
//
// Little k (kara_short): the segments are so short that the epilogue, not the
// MMAs, sets the pace, and the slots of all tiles, written and read back by the
// fold kernel, would go through memory (16384 x 256 x 16384, S = 6: 4.5 ms, 12 GB
// of slots).  There C tiles are 256 x 128: with 32 columns a thread the sums T
// and N_g both fit the registers, the segments interleave (P_1, P_2, N_3, P_3,
// N_4, ..), D_g = T + N_g goes to the CTA's own slots once (64 KiB each, 58 MB
// over all CTAs at S = 6: they stay in L2), and the thread folds its own D_g at
// the end of the tile, while four windows of 128 columns let the MMAs run on.
//
// The tiles of the last, partly filled wave are cut by segments, and by ranges
// of k where that is not enough to fill it: a work unit is then part of a
// tile's list over part of k and leaves every segment's own sums in a slot,
// which the fold kernel combines.
#include <cuda_runtime.h>

#include <cstdint>

#include "mxm_internal.h"
#include "ozaki_fold.cuh"
#include "ptx.cuh"

namespace mxm {
namespace {

constexpr int kThreads = 640;   // warp 0 copies, warp 1 issues (rank 0) or relays (rank 1),
                                // warps 4-19 run the epilogue
constexpr int kEpiWarps = 16;
constexpr int kSlots = 7;       // ring of operand tiles: A and B alternate
// columns of a C tile and of an accumulator window, windows, and columns of the
// tile per epilogue warp of the two forms
template <bool kShort>
struct Form {
  static constexpr int kN = kShort ? 128 : 256, kBufs = kShort ? 4 : 2, kCPW = kShort ? 32 : 64;
  static constexpr int kBBytes = kShort ? kOzTileBytes / 2 : kOzTileBytes;
  static constexpr int kSlotVec = kOzTileRows * kN / 4;  // int4 of a segment's sums of one CTA
};
constexpr uint32_t kTmemCols = 512;
constexpr int kMmas = kOzTileK / 16;
constexpr int kFoldCols = 256, kFoldVec = kOzTileRows * kFoldCols / 4;  // the fold kernel's tiles
constexpr int kMaxProducts = 40, kMaxSegs = 20, kMaxS = kKaraMaxSlices;

// The products of a tile in order, and the segments they form.
struct KaraProg {
  int nseg;
  uint8_t pa[kMaxProducts], pb[kMaxProducts];  // planes of A and B
  uint8_t end[kMaxSegs];    // segment i: products [end[i - 1], end[i])
  uint8_t g[kMaxSegs];      // N_g: g; the square P_s: kSquare + s
  uint8_t part[kMaxSegs + 1];  // units of a cut tile: segments [part[i], part[i + 1])
};
constexpr int kSquare = 64;

struct KaraArgs {
  const uint8_t* aslices;
  const uint8_t* bslices;
  const uint64_t* rowbits;
  const uint64_t* colbits;
  double* C;
  int4* full_scratch;   // per whole tile and rank: S slots, D_g in slot g - 2
  int4* cut_scratch;    // per cut tile, rank and k range: 2 S - 2 slots, N_g in g - 3,
                        // P_s in S - 2 + s
  int64_t m, n;
  int Mt, Nt, Kt, Mp, Np;  // Mp, Np: C tiles down and across
  int tiles, full_tiles;  // 256 x 256 C tiles; those done whole
  int raster;
  int S, beta, eoff, gx;
  int win_p, win_n;     // k-blocks per window: squares, the rest
  int last_mmas;        // MMAs of the last k-block
  int parts, ranges;    // a cut tile: units along its segments, ranges of k
  KaraProg prog;
};

struct __align__(1024) KaraSmem {
  uint8_t slot[kSlots][kOzTileBytes];
  uint64_t full[kSlots], empty[kSlots];
  uint64_t accfull[4], accempty[4];
  uint32_t tmem_base;
  int abort_flag;
};
constexpr size_t kSmemBytes = sizeof(KaraSmem) + 1024;
static_assert(kSmemBytes <= 232448, "shared memory");

struct KUnit {
  int tm, tn;   // C tile
  int s0, s1;   // segments
  int kb0, kb1; // k-blocks
  int cut;      // a cut tile: its index (cut tile, k range), else -1
  int tile;     // index of the tile in the walk
};
// C tile t of the walk (tile_coords in 32 bits).
__device__ __forceinline__ void kara_coords(const KaraArgs& a, int t, int& tm, int& tn) {
  const int grp = t / (a.raster * a.Np), first = grp * a.raster;
  const int gsz = a.Mp - first < a.raster ? a.Mp - first : a.raster;
  const int in = t - first * a.Np;
  tn = in / gsz;
  tm = first + in - tn * gsz;
}
__device__ __forceinline__ int kunits(const KaraArgs& a) {
  return a.full_tiles + (a.tiles - a.full_tiles) * a.parts * a.ranges;
}
__device__ __forceinline__ KUnit kunit(const KaraArgs& a, int u) {
  KUnit k;
  int t = u;
  if (u < a.full_tiles) {
    k.s0 = 0;
    k.s1 = a.prog.nseg;
    k.kb0 = 0;
    k.kb1 = a.Kt;
    k.cut = -1;
  } else {
    const int v = u - a.full_tiles;
    k.cut = v / a.parts;
    const int p = v - k.cut * a.parts, c = k.cut / a.ranges, q = k.cut - c * a.ranges;
    t = a.full_tiles + c;
    k.kb0 = static_cast<int>(static_cast<int64_t>(a.Kt) * q / a.ranges);
    k.kb1 = static_cast<int>(static_cast<int64_t>(a.Kt) * (q + 1) / a.ranges);
    k.s0 = a.prog.part[p];
    k.s1 = a.prog.part[p + 1];
  }
  k.tile = t;
  kara_coords(a, t, k.tm, k.tn);
  return k;
}
__device__ __forceinline__ int seg_begin(const KaraArgs& a, int s) {
  return s > 0 ? a.prog.end[s - 1] : 0;
}

struct KRing {
  int slot = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void advance() {
    if (++slot == kSlots) {
      slot = 0;
      phase ^= 1u;
    }
  }
};

// Fold the diagonals d[0] = D_{S+1}, .., d[S-2] = D_3, then d2 = D_2, of four
// neighbouring elements in the order of step 4 (exact int64 partial for
// g >= gx, FP64 additions after).  Straight-line over the longest list (D_2
// apart: indexed by S it would put the list into local memory); the bounds
// are uniform.
// Sum: int, or long long where a D_g may pass 2^31.
template <typename Sum, int kLen>
__device__ __forceinline__ void fold_columns(const Sum (&d)[kLen][4], const Sum (&d2)[4],
                                             int S, int beta, int gx, double (&out)[4]) {
  long long y[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) y[c] = d[0][c];  // diagonal S + 1 is always exact
  auto exact = [&](const Sum (&v)[4], int sh) {
#pragma unroll
    for (int c = 0; c < 4; ++c) y[c] = add_shifted(y[c], v[c], sh);
  };
#pragma unroll
  for (int i = 1; i < kLen; ++i)
    if (i <= S - 2 && i <= S + 1 - gx) exact(d[i], beta * i);  // uniform
  if (gx <= 2) exact(d2, beta * (S - 1));
#pragma unroll
  for (int c = 0; c < 4; ++c) out[c] = i64_pow2(y[c], -beta * (S + 1));
#pragma unroll
  for (int i = 1; i < kLen; ++i) {
    const int g = S + 1 - i;
    if (g >= 3 && g < gx) {  // uniform
#pragma unroll
      for (int c = 0; c < 4; ++c) out[c] = __dadd_rn(out[c], sum_pow2(d[i][c], -beta * g));
    }
  }
  if (gx > 2) {
#pragma unroll
    for (int c = 0; c < 4; ++c) out[c] = __dadd_rn(out[c], sum_pow2(d2[c], -beta * 2));
  }
}

// Slot accesses (through L2), in program order.
__device__ __forceinline__ int4 ld_cg4(const int4* p) {
  int4 v;
  asm volatile("ld.global.cg.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ void st_cg4(int4* p, const int4& v) {
  asm volatile("st.global.cg.v4.s32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}

// Four consecutive doubles of C, 32-byte aligned: one whole sector.
__device__ __forceinline__ void store4(double* p, const double (&v)[4]) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]),
               "d"(v[2]), "d"(v[3])
               : "memory");
}

template <bool kShort>
__global__ void __launch_bounds__(kThreads, 1)
    oz_kara_kernel(const __grid_constant__ KaraArgs a, int* __restrict__ status) {
  using F = Form<kShort>;
  constexpr int kN = F::kN, kBufs = F::kBufs, kCPW = F::kCPW;
  extern __shared__ uint8_t smem_raw[];
  KaraSmem& sm = *reinterpret_cast<KaraSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_cta_rank();
  const bool leader = rank == 0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&sm.full[i], leader ? 2 : 1);  // rank 0: + the relay's arrival
      mbar_init(&sm.empty[i], 1);
    }
    for (int i = 0; i < kBufs; ++i) {
      mbar_init(&sm.accfull[i], 1);
      mbar_init(&sm.accempty[i], 2 * kEpiWarps);
    }
    sm.abort_flag = 0;
    fence_mbar_init();
  }
  cluster_sync_all();  // barriers initialised before any peer arrives
  if (warp == 1) {
    tmem_alloc_pair(&sm.tmem_base, kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;
  volatile int* abort_flag = &sm.abort_flag;
  follow_grid();
  release_next();
  const int nunits = kunits(a);
  const int unit0 = blockIdx.x >> 1, unit_step = gridDim.x >> 1;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;" ::: "memory");
    if (warp == 0 && lane == 0) {
      // ------------------------------------------------ producer (bulk copies)
      KRing r;
      bool ok = true;
      auto load = [&](const uint8_t* src, uint32_t bytes) {  // nullptr: nothing there (past the last tile)
        if (!mbar_wait_bounded(&sm.empty[r.slot], r.phase ^ 1u, abort_flag, status)) return false;
        if (src != nullptr) {
          mbar_arrive_expect_tx(&sm.full[r.slot], bytes);
          bulk_g2s(sm.slot[r.slot], src, bytes, &sm.full[r.slot]);
        } else {
          mbar_arrive(&sm.full[r.slot]);
        }
        r.advance();
        return true;
      };
      const size_t a_plane = static_cast<size_t>(a.Mt) * a.Kt * kOzTileBytes;
      const size_t b_plane = static_cast<size_t>(a.Nt) * a.Kt * kOzTileBytes;
      for (int u = unit0; u < nunits && ok; u += unit_step) {
        const KUnit k = kunit(a, u);
        const int ta = 2 * k.tm + static_cast<int>(rank);
        const int tb = kShort ? k.tn : 2 * k.tn + static_cast<int>(rank);
        const bool alive = ta < a.Mt, blive = tb < a.Nt;
        const uint8_t* a0 = a.aslices + static_cast<size_t>(ta) * a.Kt * kOzTileBytes;
        // short: the CTA's half of the tile (oz_chunk_offset_halves)
        const uint8_t* b0 = a.bslices + static_cast<size_t>(tb) * a.Kt * kOzTileBytes +
                            (kShort ? rank * F::kBBytes : 0);
        const int p1 = seg_begin(a, k.s1);
        for (int p = seg_begin(a, k.s0); p < p1 && ok; ++p) {
          const uint8_t* ap = a0 + a.prog.pa[p] * a_plane;
          const uint8_t* bp = b0 + a.prog.pb[p] * b_plane;
          MXM_BOUNDS(!alive || in_range(ap, a.Kt * kOzTileBytes, a.aslices,
                                        a.aslices + a_plane * kara_planes(a.S)), status);
          MXM_BOUNDS(!blive || in_range(bp, (a.Kt - 1) * kOzTileBytes + F::kBBytes, a.bslices,
                                        a.bslices + b_plane * kara_planes(a.S)), status);
          for (int kb = k.kb0; kb < k.kb1 && ok; ++kb)
            ok = load(alive ? ap + static_cast<size_t>(kb) * kOzTileBytes : nullptr, kOzTileBytes) &&
                 load(blive ? bp + static_cast<size_t>(kb) * kOzTileBytes : nullptr, F::kBBytes);
        }
      }
      // tail: wait until every slot is released, so that no copy or commit
      // lands after the block has exited
      for (int i = 0; i < kSlots; ++i) {
        if (!mbar_wait_bounded(&sm.empty[r.slot], r.phase ^ 1u, abort_flag, status)) break;
        r.advance();
      }
    } else if (!leader && warp == 1 && lane == 0) {
      // ------------------------------------------------ relay (rank 1): a tile of
      // this CTA has landed -> arrive on the same slot's full barrier of rank 0
      KRing r;
      bool ok = true;
      for (int u = unit0; u < nunits && ok; u += unit_step) {
        const KUnit k = kunit(a, u);
        const int loads = 2 * (k.kb1 - k.kb0) * (seg_begin(a, k.s1) - seg_begin(a, k.s0));
        for (int i = 0; i < loads; ++i) {
          if (!mbar_wait_bounded(&sm.full[r.slot], r.phase, abort_flag, status)) {
            ok = false;
            break;
          }
          mbar_arrive_remote_release(smem_in_cta(&sm.full[r.slot], 0));
          r.advance();
        }
      }
    } else if (leader && warp == 1 && lane == 0) {
      // ------------------------------------------------ MMA issuer
      const uint32_t idesc = idesc_bf16_f32(256, kN);
      const uint64_t desc0 = sw128_kmajor_desc(smem_u32(sm.slot[0]));
      KRing r;
      uint32_t win = 0;  // windows started
      bool ok = true;
      bool seen_a = false, seen_b = false;  // the next slots were seen full (mbar_test)
      auto wait_full = [&](bool& seen) -> bool {
        if (seen) {
          seen = false;
          fence_acquire_cluster_shared();
          return true;
        }
        return mbar_wait_bounded<false, true>(&sm.full[r.slot], r.phase, abort_flag, status);
      };
      for (int u = unit0; u < nunits && ok; u += unit_step) {
        const KUnit k = kunit(a, u);
        for (int s = k.s0; s < k.s1 && ok; ++s) {
          const int window = a.prog.g[s] >= kSquare ? a.win_p : a.win_n;
          const int steps = (k.kb1 - k.kb0) * (a.prog.end[s] - seg_begin(a, s));
          int cnt = 0, kb = k.kb0;
          for (int st = 0; st < steps; ++st) {
            if (!wait_full(seen_a)) {
              ok = false;
              break;
            }
            const int sa = r.slot;
            r.advance();
            if (!wait_full(seen_b)) {
              ok = false;
              break;
            }
            const int sb = r.slot;
            r.advance();
            const int buf = win % kBufs;
            if (cnt == 0 && win >= kBufs &&  // a window starts: its buffer must have been drained
                !mbar_wait_bounded<false, true>(&sm.accempty[buf], (win / kBufs - 1u) & 1u,
                                                abort_flag, status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t da = desc0 + static_cast<uint64_t>(sa) * (kOzTileBytes >> 4);
            const uint64_t db = desc0 + static_cast<uint64_t>(sb) * (kOzTileBytes >> 4);
            const uint32_t d = tmem + static_cast<uint32_t>(buf * kN);
            const int nmma = kb == a.Kt - 1 ? a.last_mmas : kMmas;
            const uint32_t acc0 = cnt > 0 ? 1u : 0u;
            KRing nx = r;
#pragma unroll
            for (int kk = 0; kk < kMmas; ++kk) {
              const uint64_t off =
                  static_cast<uint64_t>((kk >> 2) * (kOzAtomBytes >> 4) + (kk & 3) * 2);
              const uint64_t boff =  // short: atoms of 64 rows, 8 KiB apart
                  kShort ? static_cast<uint64_t>((kk >> 2) * (kOzAtomBytes >> 5) + (kk & 3) * 2) : off;
              if (kk < nmma) mma_bf16_ss_pair(d, da + off, db + boff, idesc, kk > 0 ? 1u : acc0);
              if (kk == kMmas / 2 - 1) {  // half-way: the slots the next waits are on
                seen_a = mbar_test<true>(&sm.full[nx.slot], nx.phase);
                nx.advance();
                seen_b = mbar_test<true>(&sm.full[nx.slot], nx.phase);
              }
            }
            mma_commit_pair(&sm.empty[sa], static_cast<uint16_t>(0x3));
            mma_commit_pair(&sm.empty[sb], static_cast<uint16_t>(0x3));
            if (++cnt == window || st + 1 == steps) {
              mma_commit_pair(&sm.accfull[buf], static_cast<uint16_t>(0x3));
              ++win;
              cnt = 0;
            }
            if (++kb == k.kb1) kb = k.kb0;
          }
        }
      }
    }
  } else {
    // ------------------------------------------------ epilogue (16 warps)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;" ::: "memory");
    const int quarter = warp & 3;           // TMEM lanes this warp may access
    const int cg = (warp - 4) >> 2;         // which 64 columns of the tile
    const int row_in_tile = quarter * 32 + lane;
    const uint32_t t_lane = tmem + (static_cast<uint32_t>(quarter * 32) << 16) +
                            static_cast<uint32_t>(cg * kCPW);
    const int S = a.S;
    // this thread's 4-column groups: group c of a slot at + c * 128
    const int own = cg * (kCPW / 4) * kOzTileRows + row_in_tile;
    constexpr int kSlotVec = F::kSlotVec;
    uint32_t win = 0;  // windows drained
    bool ok = true;
    int D[kCPW];                   // a segment's sums; short: T
    int Ng[kShort ? kCPW : 1];     // short: N_g

    auto wait_window = [&]() -> bool {
      if (!mbar_wait_bounded(&sm.accfull[win % kBufs], (win / kBufs) & 1u, abort_flag, status))
        return false;
      tc_fence_after();
      return true;
    };
    auto free_window = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        uint64_t* const empty = &sm.accempty[win % kBufs];
        if (!leader)
          mbar_arrive_remote_release(smem_in_cta(empty, 0));  // the issuer is in rank 0
        else
          mbar_arrive(empty);
      }
      ++win;
    };
    // every window of segment s added into X
    auto drain = [&](int s, int kblocks, int (&X)[kCPW]) -> bool {
      const int window = a.prog.g[s] >= kSquare ? a.win_p : a.win_n;
      const int steps = kblocks * (a.prog.end[s] - seg_begin(a, s));
      for (int st = 0; st < steps; st += window) {
        if (!wait_window()) return false;
#pragma unroll
        for (int h = 0; h < kCPW / 16; ++h) {
          uint32_t r[16];
          tmem_ld16(t_lane + static_cast<uint32_t>((win % kBufs) * kN + h * 16), r);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) X[h * 16 + i] += __float2int_rz(__uint_as_float(r[i]));
        }
        free_window();
      }
      return true;
    };
    auto put = [&](int4* slot) {
#pragma unroll
      for (int c = 0; c < kCPW / 4; ++c)
        st_cg4(slot + own + c * kOzTileRows,
               make_int4(D[4 * c], D[4 * c + 1], D[4 * c + 2], D[4 * c + 3]));
    };
    auto get = [&](const int4* slot) {  // this thread's own stores
#pragma unroll
      for (int c = 0; c < kCPW / 4; ++c) {
        const int4 v = ld_cg4(slot + own + c * kOzTileRows);
        D[4 * c] = v.x;
        D[4 * c + 1] = v.y;
        D[4 * c + 2] = v.z;
        D[4 * c + 3] = v.w;
      }
    };

    for (int u = unit0; u < nunits && ok; u += unit_step) {
      const KUnit k = kunit(a, u);
      const int64_t row0 = (2 * static_cast<int64_t>(k.tm) + rank) * kOzTileRows;
      const int64_t col0 = static_cast<int64_t>(k.tn) * kN + cg * kCPW;
      // a part of the tile outside C (warp-uniform): its windows are drained only
      const bool keep = row0 + quarter * 32 < a.m && col0 < a.n;
      if constexpr (kShort) {
        // ---------------- short: P_1, P_2, N_3, P_3, .., P_{S-1}, N_S, N_{S+1}
        int4* const base = a.full_scratch + static_cast<size_t>(blockIdx.x) * S * kSlotVec;
#pragma unroll
        for (int i = 0; i < kCPW; ++i) D[i] = 0;
        for (int s = 0; s < k.s1 && ok; ++s) {
          const int g = a.prog.g[s];
          if (g >= kSquare) {
            ok = drain(s, a.Kt, D);
            if (ok && keep && g == kSquare + 1) {
#pragma unroll
              for (int c = 0; c < kCPW / 4; ++c)
                st_cg4(base + own + c * kOzTileRows,
                       make_int4(D[4 * c], D[4 * c + 1], D[4 * c + 2], D[4 * c + 3]));
            }
          } else {
#pragma unroll
            for (int i = 0; i < kCPW; ++i) Ng[i] = 0;
            ok = drain(s, a.Kt, Ng);
            if (ok && keep) {
              int4* const slot = base + static_cast<size_t>(g - 2) * kSlotVec;
#pragma unroll
              for (int c = 0; c < kCPW / 4; ++c)
                st_cg4(slot + own + c * kOzTileRows,
                       make_int4(D[4 * c] + Ng[4 * c], D[4 * c + 1] + Ng[4 * c + 1],
                                 D[4 * c + 2] + Ng[4 * c + 2], D[4 * c + 3] + Ng[4 * c + 3]));
            }
          }
        }
        if (!ok) break;
        if (!keep) continue;
        const int64_t row = row0 + row_in_tile;
        const bool row_ok = row < a.m;
        const int er = row_ok ? exponent_from_absbits(a.rowbits[row]) + a.eoff : 0;
        // lane l holds the exponent of this warp's column l
        const int64_t lcol = col0 + lane;
        const int ec = lcol < a.n ? exponent_from_absbits(__ldg(a.colbits + lcol)) : 0;
        double* const crow = a.C + (row_ok ? row : 0) * a.n;
        const bool vec = (a.n & 3) == 0 && (reinterpret_cast<uintptr_t>(a.C) & 31) == 0;
        const int groups = a.n - col0 >= kCPW ? kCPW / 4 : static_cast<int>((a.n - col0 + 3) / 4);
        // a group's slots are read one group ahead (T and N_g are dead here)
        int4 nx[kKaraShortSlices - 1], nx2;
        auto read = [&](int c) {
          const int4* p = base + own + c * kOzTileRows;
#pragma unroll
          for (int i = 0; i < kKaraShortSlices - 1; ++i)
            if (i < S - 1) nx[i] = __ldcg(p + static_cast<size_t>(S - 1 - i) * kSlotVec);
          nx2 = __ldcg(p);  // D_2 = P_1
        };
#pragma unroll
        for (int i = 0; i < kKaraShortSlices - 1; ++i) nx[i] = make_int4(0, 0, 0, 0);
        read(0);
#pragma unroll 1
        for (int c = 0; c < groups; ++c) {
          int d[kKaraShortSlices - 1][4];
          const int d2[4] = {nx2.x, nx2.y, nx2.z, nx2.w};
#pragma unroll
          for (int i = 0; i < kKaraShortSlices - 1; ++i) {
            d[i][0] = nx[i].x;
            d[i][1] = nx[i].y;
            d[i][2] = nx[i].z;
            d[i][3] = nx[i].w;
          }
          if (c + 1 < groups) read(c + 1);
#pragma unroll
          for (int j = 0; j < 4; ++j) d[0][j] -= d2[j];  // the pair (1, S) was taken directly
          double out[4];
          fold_columns(d, d2, S, a.beta, a.gx, out);
          const int64_t col = col0 + 4 * c;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            out[j] = scale_by(out[j], er + __shfl_sync(0xFFFFFFFFu, ec, 4 * c + j));
          if (!row_ok) continue;
          if (vec && col + 4 <= a.n) {
            store4(crow + col, out);
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (col + j < a.n) crow[col + j] = out[j];
          }
        }
      } else {
        int4* const base =
            k.cut < 0
                ? a.full_scratch + (static_cast<size_t>(k.tile) * 2 + rank) * S * kSlotVec
                : a.cut_scratch + (static_cast<size_t>(k.cut) * 2 + rank) * (2 * S - 2) * kSlotVec;
        for (int s = k.s0; s < k.s1 && ok; ++s) {
          const int g = a.prog.g[s];
          const bool square = g >= kSquare;
          const int sq = g - kSquare;
          int4* const slot =
              base + static_cast<size_t>(k.cut >= 0 ? (square ? S - 2 + sq : g - 3)
                                                    : (square ? sq - 1 : g - 2)) * kSlotVec;
          if (k.cut < 0 && !square) {
            if (keep) get(slot);  // T_g; in flight until the first window is read
          } else if (k.cut >= 0 || sq == 1) {
#pragma unroll
            for (int i = 0; i < kCPW; ++i) D[i] = 0;
          }
          ok = drain(s, k.kb1 - k.kb0, D);
          if (!ok || !keep) continue;
          put(slot);
          // D_{S+1} starts from T_S as well (the fold takes P_1 = D_2 out of it)
          if (k.cut < 0 && sq == S - 1) put(slot + kSlotVec);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA leaves (nor frees its tensor memory) while the other may
  // still arrive on its barriers or run MMAs into it
  cluster_sync_all();
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, kTmemCols);
}

__device__ __forceinline__ void add4(int (&v)[4], const int4& x) {
  v[0] += x.x;
  v[1] += x.y;
  v[2] += x.z;
  v[3] += x.w;
}

// Step 4 from the slots: a thread takes four neighbouring columns of one row,
// with all its slot reads in flight at once.  Bound by HBM (4 S bytes read and
// 8 written per element; S = 7 at 8192^2: 2.4 GB).  kCut: the tiles cut into
// units (2 S - 2 slots per k range), else the whole tiles (S slots).
// Sum: the type of D_g; every k range's part of it fits int32.
constexpr int kFoldThreads = 128;
template <bool kCut, typename Sum>
__global__ void __launch_bounds__(kFoldThreads) oz_kara_fold_kernel(
    const __grid_constant__ KaraArgs a, int part0) {
  constexpr int kSlotVec = kFoldVec;
  const int S = a.S;
  follow_grid();
  release_next();
  const int part = part0 + blockIdx.y;  // (tile, rank) among the kind's tiles
  const int t = (kCut ? a.full_tiles : 0) + (part >> 1), rank = part & 1;
  int tm, tn;
  kara_coords(a, t, tm, tn);
  const int v = blockIdx.x * kFoldThreads + threadIdx.x;  // column group v / 128, row v % 128
  const int64_t row = (2 * static_cast<int64_t>(tm) + rank) * kOzTileRows + (v & 127);
  const int64_t col = static_cast<int64_t>(tn) * kFoldCols + 4 * (v >> 7);
  if (row >= a.m || col >= a.n) return;
  Sum d[kMaxS - 1][4], d2[4];  // D_{S+1} .. D_3, and D_2
  if constexpr (kCut) {
    // N_g and P_s; T_g = P_1 + .. + P_{g-1}, D_g = T_g + N_g (and T_S for
    // D_{S+1}), D_2 = P_1.  With int32 D_g the k ranges' N_g and P_s are
    // added first, with 64-bit ones each range's D_g are.
    constexpr bool kWide = sizeof(Sum) == 8;
    const size_t range = 2 * static_cast<size_t>(2 * S - 2) * kSlotVec;
    const int4* p = after_follow(a.cut_scratch) + static_cast<size_t>(part >> 1) * a.ranges * range +
                    static_cast<size_t>(rank) * (2 * S - 2) * kSlotVec + v;
    int ng[kMaxS - 1][4], sq[kMaxS - 1][4];  // N_{S+1} .. N_3, P_{S-1} .. P_1
    auto clear = [&]() {
#pragma unroll
      for (int i = 0; i < kMaxS - 1; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) ng[i][j] = sq[i][j] = 0;
    };
    auto read = [&]() {
      int4 x[kMaxS - 1], y[kMaxS - 1];
#pragma unroll
      for (int i = 0; i < kMaxS - 1; ++i)
        if (i < S - 1) {
          x[i] = __ldcs(p + static_cast<size_t>(S - 2 - i) * kSlotVec);
          y[i] = __ldcs(p + static_cast<size_t>(2 * S - 3 - i) * kSlotVec);
        }
#pragma unroll
      for (int i = 0; i < kMaxS - 1; ++i)
        if (i < S - 1) {
          add4(ng[i], x[i]);
          add4(sq[i], y[i]);
        }
      p += range;
    };
    auto combine = [&]() {
      int T[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        T[j] = sq[kMaxS - 2][j];  // up from P_1 (zeros before it): sq[i - 1] = P_{S-i}
        if (S == kMaxS) d2[j] += T[j];
      }
#pragma unroll
      for (int i = kMaxS - 2; i >= 1; --i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          T[j] += sq[i - 1][j];
          if (i == S - 1) d2[j] += T[j];  // P_1 alone
          if (i < S - 1) d[i][j] += ng[i][j] + T[j];
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) d[0][j] += ng[0][j] + T[j];
    };
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      d2[j] = 0;
#pragma unroll
      for (int i = 0; i < kMaxS - 1; ++i) d[i][j] = 0;
    }
    clear();
#pragma unroll 1
    for (int r = 0; r < a.ranges; ++r) {
      if (kWide && r > 0) clear();
      read();
      if (kWide) combine();
    }
    if (!kWide) combine();
  } else {
    const int4* p =
        after_follow(a.full_scratch) + static_cast<size_t>(part) * S * kSlotVec + v;
#pragma unroll
    for (int i = 0; i < kMaxS - 1; ++i) {
      const int4 x = i < S - 1 ? __ldcs(p + static_cast<size_t>(S - 1 - i) * kSlotVec)
                               : make_int4(0, 0, 0, 0);
      d[i][0] = x.x;
      d[i][1] = x.y;
      d[i][2] = x.z;
      d[i][3] = x.w;
    }
    const int4 x = __ldcs(p);
    d2[0] = x.x;
    d2[1] = x.y;
    d2[2] = x.z;
    d2[3] = x.w;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) d[0][j] -= d2[j];  // the pair (1, S) was taken directly
  double out[4];
  fold_columns(d, d2, S, a.beta, a.gx, out);
  const int er = exponent_from_absbits(__ldg(a.rowbits + row)) + a.eoff;
  double* const c = a.C + row * a.n + col;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (col + j < a.n) out[j] = scale_by(out[j], er + exponent_from_absbits(__ldg(a.colbits + col + j)));
  if ((a.n & 3) == 0 && (reinterpret_cast<uintptr_t>(a.C) & 31) == 0) {
    store4(c, out);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (col + j < a.n) c[j] = out[j];
  }
}

// The products and segments of S slices: the squares, then the N_g; inter: P_1,
// then each square with the N_g that follows it.
void build_prog(int S, bool inter, KaraProg& pr) {
  int np = 0, ns = 0;
  auto square = [&](int s) {
    pr.pa[np] = pr.pb[np] = static_cast<uint8_t>(s - 1);
    ++np;
    pr.end[ns] = static_cast<uint8_t>(np);
    pr.g[ns++] = static_cast<uint8_t>(kSquare + s);
  };
  auto ndiag = [&](int g) {
    for (int s = 1; s < g - s; ++s) {
      const int t = g - s;
      if (s == 1 && t == S) {  // directly: A_1 B_S + A_S B_1
        pr.pa[np] = 0;
        pr.pb[np++] = static_cast<uint8_t>(S - 1);
        pr.pa[np] = static_cast<uint8_t>(S - 1);
        pr.pb[np++] = 0;
      } else {
        pr.pa[np] = pr.pb[np] = static_cast<uint8_t>(kara_pair_plane(S, s, t));
        ++np;
      }
    }
    pr.end[ns] = static_cast<uint8_t>(np);
    pr.g[ns++] = static_cast<uint8_t>(g);
  };
  if (inter) {
    square(1);
    for (int s = 2; s <= S - 1; ++s) {
      square(s);
      ndiag(s + 1);
    }
    ndiag(S + 1);
  } else {
    for (int s = 1; s <= S - 1; ++s) square(s);
    for (int g = 3; g <= S + 1; ++g) ndiag(g);
  }
  pr.nseg = ns;
}

// Boundaries of `parts` runs of segments with nearly equal numbers of
// products; returns the largest run's products.
int cut_segments(const KaraProg& pr, int parts, uint8_t* part) {
  const int total = pr.end[pr.nseg - 1];
  int at = 0, worst = 0;
  part[0] = 0;
  for (int i = 1; i <= parts; ++i) {
    const int want = (total * i + parts / 2) / parts, from = at > 0 ? pr.end[at - 1] : 0;
    ++at;  // at least one segment each, and enough left for the others
    while (at < pr.nseg - (parts - i) && (i == parts || pr.end[at - 1] < want)) ++at;
    part[i] = static_cast<uint8_t>(at);
    if (pr.end[at - 1] - from > worst) worst = pr.end[at - 1] - from;
  }
  return worst;
}

// How the `rest` tiles of the last wave are cut into units (parts along the
// segments times ranges of k), by an estimate in k-blocks of one product (0.53
// us): the waves of units, each with its longest run of products, 2 per
// segment for its slot, and the fold's reading of the slots.  false: whole.
// Never fewer ranges than keep a range's sums in int32.
bool choose_cut(const OzakiDims& d, int64_t rest, int64_t pairs, KaraArgs& a) {
  const int least = kara_min_ranges(d);
  const int total = a.prog.end[a.prog.nseg - 1], nslots = 2 * d.S - 2;
  const double slot_read = 0.25;  // 2 x 128 KiB at about 2 TB/s
  double best = static_cast<double>(d.Kt) * total + 2.0 * a.prog.nseg + slot_read * rest * d.S;
  if (least > 1) best = 1e30;
  int best_parts = 1, best_ranges = 1;
  uint8_t part[kMaxSegs + 1];
  for (int parts = 1; parts <= a.prog.nseg; ++parts) {
    const int worst = cut_segments(a.prog, parts, part);
    const int segs = (a.prog.nseg + parts - 1) / parts;
    for (int ranges = least; ranges <= kara_max_ranges(d); ++ranges) {
      if (static_cast<size_t>(rest * ranges * nslots) > kara_cut_slots(d)) break;
      const int64_t waves = (rest * parts * ranges + pairs - 1) / pairs;
      const double cost = waves * (static_cast<double>((d.Kt + ranges - 1) / ranges) * worst +
                                   2.0 * segs) +
                          slot_read * rest * ranges * nslots;
      if (cost < best) {
        best = cost;
        best_parts = parts;
        best_ranges = ranges;
      }
    }
  }
  if (best_parts * best_ranges == 1) return false;
  a.parts = best_parts;
  a.ranges = best_ranges;
  cut_segments(a.prog, best_parts, a.prog.part);
  return true;
}

}  // namespace

cudaError_t launch_ozaki_kara(const uint8_t* aslices, const uint8_t* bslices,
                              const uint64_t* rowbits, const uint64_t* colbits, double* C,
                              const OzakiDims& d, uint8_t* scratch, int* status,
                              cudaStream_t s) {
  KaraArgs a;
  a.aslices = aslices;
  a.bslices = bslices;
  a.rowbits = rowbits;
  a.colbits = colbits;
  a.C = C;
  a.m = d.m;
  a.n = d.n;
  a.Mt = static_cast<int>(d.Mt);
  a.Nt = static_cast<int>(d.Nt);
  a.Kt = static_cast<int>(d.Kt);
  a.S = d.S;
  a.beta = d.beta;
  a.eoff = d.rn ? 2 : 0;
  a.gx = ozaki_exact_from(d.S, d.beta, d.Kt);
  a.win_p = ozaki_window_stages(d.beta, d.rn != 0);
  a.win_n = kara_window_stages(d);
  const int64_t klast = d.k - (d.Kt - 1) * kOzTileK;
  a.last_mmas = static_cast<int>((klast + 15) / 16);
  const bool is_short = d.kara == 2;
  const int64_t Mp = (d.Mt + 1) / 2;
  a.Mp = static_cast<int>(Mp);
  a.Np = static_cast<int>(is_short ? d.Nt : (d.Nt + 1) / 2);
  a.raster = static_cast<int>(d.raster < Mp ? (d.raster > 0 ? d.raster : kDefaultRaster) : Mp);
  build_prog(d.S, is_short, a.prog);
  const auto kern = is_short ? oz_kara_kernel<true> : oz_kara_kernel<false>;
  static PerDevice limit[2], held[2];
  cudaError_t e = allow_smem(limit[is_short], kern, kSmemBytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(2, 1, 1);
  int clusters = 0;
  e = held[is_short].get(&clusters, [&](int* v) {
    return cudaOccupancyMaxActiveClusters(v, kern, &cfg);
  });
  if (e != cudaSuccess) return e;
  if (clusters < 1) return cudaErrorLaunchOutOfResources;
  const int64_t pairs = clusters < kKaraPairs ? clusters : kKaraPairs;
  // whole waves of tiles, then the rest, cut where that is shorter
  const int64_t tiles = static_cast<int64_t>(a.Mp) * a.Np;
  a.tiles = static_cast<int>(tiles);
  const bool wide = kara_min_ranges(d) > 1;  // every tile is cut along k
  const int64_t rest = is_short ? 0 : wide ? tiles : tiles % pairs;
  a.full_tiles = static_cast<int>(tiles - rest);
  a.parts = a.ranges = 1;
  if (rest > 0 && !choose_cut(d, rest, pairs, a)) a.full_tiles = a.tiles;
  a.full_scratch = reinterpret_cast<int4*>(scratch);
  a.cut_scratch = a.full_scratch + static_cast<size_t>(a.full_tiles) * 2 * d.S * kFoldVec;
  const int64_t units = a.full_tiles + (tiles - a.full_tiles) * a.parts * a.ranges;
  const int64_t use = units < pairs ? units : pairs;
  cfg.gridDim = dim3(static_cast<unsigned>(2 * use), 1, 1);
  cfg.numAttrs = d.chain ? 2 : 1;
  e = cudaLaunchKernelEx(&cfg, kern, a, status);
  if (e != cudaSuccess || is_short) return e;
  // (tile, rank) parts on the y axis of the grid, at most kFoldParts per launch
  constexpr int64_t kFoldParts = 32768;
  auto fold = [&](auto kern, int64_t parts) {
    for (int64_t p0 = 0; p0 < parts && e == cudaSuccess; p0 += kFoldParts) {
      const int64_t now = parts - p0 < kFoldParts ? parts - p0 : kFoldParts;
      e = launch_chained(d.chain, kern,
                         dim3(kFoldVec / kFoldThreads, static_cast<unsigned>(now)), kFoldThreads,
                         0, s, a, static_cast<int>(p0));
    }
  };
  fold(oz_kara_fold_kernel<false, int>, 2 * static_cast<int64_t>(a.full_tiles));
  const int64_t cut = 2 * (tiles - a.full_tiles);
  if (wide) fold(oz_kara_fold_kernel<true, long long>, cut);
  else fold(oz_kara_fold_kernel<true, int>, cut);
  return e;
}

}  // namespace mxm
