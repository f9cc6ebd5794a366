// f64.cu -- native FP64 product C = A.B (mod2am, Sec. 3.1) on the FP64
// tensor path (DMMA, mma.sync m16n8k4 .f64).
//
// The FP64 pipe is the limit on this GPU by far: a DMMA m16n8k4 holds an SM
// sub-partition's pipe for ~1,100 clocks, and one k step of a warp's 32 x 32
// piece of C (8 DMMAs, 2 KiB of operands) takes ~4 us.  So the operands come
// straight from the caller's arrays, one step ahead, with no packed copies
// and no shared memory, and what matters is that every sub-partition gets the
// same number of DMMAs: the paper's k-blocked rank-u update (arbb_mxm2b) is
// cut into equal shares across pieces and k.  8192^3: 1000 ms, 1.10 TFLOP/s,
// all of the DMMA probe's rate (128 x 128 tiles staged by bulk copies, whole
// tiles per CTA: 1033 ms; 2048^3: 15.7 against 19.1 ms, 256^3: 46 us against
// 615 us, where those tiles left most SMs idle).
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "mxm_internal.h"
#include "ptx.cuh"

namespace mxm {
namespace {

__device__ __forceinline__ void dmma_16x8x4(double (&d)[4], double a0, double a1, double b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k4.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
      "{%0,%1,%2,%3};"
      : "+d"(d[0]), "+d"(d[1]), "+d"(d[2]), "+d"(d[3])
      : "d"(a0), "d"(a1), "d"(b0));
}

// The live DMMA blocks of a piece (ML of its two m16 rows, NL of its four n8
// columns) as compile-time constants: a predicated-off DMMA still costs the
// pipe ~150 clocks (edge pieces ran 13-30 % longer that way), so each shape
// has its own loop.
template <typename F>
__device__ __forceinline__ void f64_with_blocks(bool two, int nlive, const F& f) {
  using C1 = std::integral_constant<int, 1>;
  using C2 = std::integral_constant<int, 2>;
  using C3 = std::integral_constant<int, 3>;
  using C4 = std::integral_constant<int, 4>;
  if (two) {
    switch (nlive) {
      case 4: f(C2{}, C4{}); break;
      case 3: f(C2{}, C3{}); break;
      case 2: f(C2{}, C2{}); break;
      default: f(C2{}, C1{}); break;
    }
  } else {
    switch (nlive) {
      case 4: f(C1{}, C4{}); break;
      case 3: f(C1{}, C3{}); break;
      case 2: f(C1{}, C2{}); break;
      default: f(C1{}, C1{}); break;
    }
  }
}

// ---------------------------------------------------------------- grouped
// Many small products of uneven sizes: the work is cut into 32 x 32 pieces
// of the C matrices (the plan's tiles), one warp each, handed out by an
// atomic cursor in the plan header (dynamic scheduling: pieces of long-k
// problems cost more).  The FP64 pipe of this GPU (~3.5 flops per clock per
// SM) is the limit, so the operands are read straight from the caller's
// arrays (L1/L2 serve the reuse) with no packed copies, and the pieces are
// small enough that padding wastes little: every product is cut at 32 rows,
// 32 columns and 4 k, and the DMMA blocks of an edge piece that lie wholly
// past the last row (16) or column (8) are not issued.  Each warp holds its
// 32 x 32 piece as 2 x 4 DMMA m16n8 accumulators and reads the fragments of
// the next k step while the current ones multiply.
constexpr int kGroupedF64Threads = 256;

__device__ __forceinline__ void load_frags(const double* __restrict__ A,
                                           const double* __restrict__ B, int64_t k, int64_t n,
                                           const int64_t (&arow)[4], const int64_t (&bcol)[4],
                                           uint32_t rmask, uint32_t cmask, int64_t kk,
                                           double (&a)[4], double (&b)[4]) {
  const bool kv = kk < k;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    a[i] = (kv && ((rmask >> i) & 1u)) ? __ldg(A + arow[i] * k + kk) : 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    b[i] = (kv && ((cmask >> i) & 1u)) ? __ldg(B + kk * n + bcol[i]) : 0.0;
}

__global__ void __launch_bounds__(kGroupedF64Threads, 2)
    f64_grouped_kernel(uint8_t* __restrict__ ws, int* __restrict__ status) {
  GroupedHeader* hdr = reinterpret_cast<GroupedHeader*>(ws);
  if (!hdr->valid) return;
  const GroupedProblem* recs = reinterpret_cast<const GroupedProblem*>(ws + kGroupedRecordsOff);
  unsigned long long* cursor = reinterpret_cast<unsigned long long*>(&hdr->cursor);
  const int64_t total = hdr->tiles;
  const int64_t count = hdr->count;
  const int lane = threadIdx.x & 31;
  const int g = lane >> 2, t4 = lane & 3;
  constexpr int T = kF64GroupedTile;
  for (;;) {
    int64_t unit = 0;
    if (lane == 0) unit = static_cast<int64_t>(atomicAdd(cursor, 1ull));
    unit = __shfl_sync(0xFFFFFFFFu, unit, 0);
    if (unit >= total) break;
    const GroupedProblem& r = recs[grouped_find(recs, count, unit, &GroupedProblem::tile_begin)];
    const int64_t local = unit - r.tile_begin;
    const int64_t tm = local / r.Nt, tn = local - (local / r.Nt) * r.Nt;
    const int64_t row0 = tm * T, col0 = tn * T;
    MXM_BOUNDS(row0 < r.m && col0 < r.n && local < r.Mt * r.Nt, status);
    const double* A = r.A;
    const double* B = r.B;
    const int64_t m = r.m, k = r.k, n = r.n;
    // this lane's A rows (mi = 0, 1; halves g, g + 8) and B columns (ni = 0..3)
    int64_t arow[4], bcol[4];
    uint32_t rmask = 0, cmask = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      arow[i] = row0 + (i >> 1) * 16 + (i & 1) * 8 + g;
      if (arow[i] < m) rmask |= 1u << i;
      bcol[i] = col0 + i * 8 + g;
      if (bcol[i] < n) cmask |= 1u << i;
    }
    double acc[2][4][4];
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
      for (int ni = 0; ni < 4; ++ni)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[mi][ni][q] = 0.0;
    // the m16 / n8 blocks holding any row / column of C (warp-uniform)
    const bool mlive1 = row0 + 16 < m;
    const int nlive = static_cast<int>((n - col0 + 7) / 8 < 4 ? (n - col0 + 7) / 8 : 4);
    double a[4], b[4], an[4], bn[4];
    load_frags(A, B, k, n, arow, bcol, rmask, cmask, t4, a, b);
    f64_with_blocks(mlive1, nlive, [&](auto ml, auto nl) {
      for (int64_t k0 = 0; k0 < k; k0 += kF64GroupedK) {
        load_frags(A, B, k, n, arow, bcol, rmask, cmask, k0 + kF64GroupedK + t4, an, bn);
#pragma unroll
        for (int mi = 0; mi < decltype(ml)::value; ++mi)
#pragma unroll
          for (int ni = 0; ni < decltype(nl)::value; ++ni)
            dmma_16x8x4(acc[mi][ni], a[2 * mi], a[2 * mi + 1], b[ni]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          a[i] = an[i];
          b[i] = bn[i];
        }
      }
    });
    // D fragment of m16n8: (g, 2 t4), (g, 2 t4 + 1), (g + 8, 2 t4), (g + 8, 2 t4 + 1)
#pragma unroll
    for (int mi = 0; mi < 2; ++mi) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t row = row0 + mi * 16 + h * 8 + g;
        if (row >= m) continue;
        double* crow = r.C + row * n;
#pragma unroll
        for (int ni = 0; ni < 4; ++ni) {
          const int64_t col = col0 + ni * 8 + 2 * t4;
          if (col < n) crow[col] = acc[mi][ni][2 * h];
          if (col + 1 < n) crow[col + 1] = acc[mi][ni][2 * h + 1];
        }
      }
    }
  }
}

// ---------------------------------------------------------------- balanced
// The product cut into equal shares of DMMA work: the C matrix in 32 x 32
// pieces, each of Ks = ceil(k / 4) steps of up to 8 DMMAs m16n8k4 (the blocks
// of an edge piece past the last row or column are not issued), walked piece
// after piece, k inside; worker i of W takes the i-th W-th of that walk,
// whatever piece it starts or ends in.  The FP64 pipe is the limit (a DMMA
// holds an SM sub-partition's for ~1,100 clocks, a step for ~4 us), so the
// operands come straight from the caller's arrays, loaded one step ahead, and
// only the balance counts: W = 1216, two warps per sub-partition of 152 SMs (a
// constant: the rounding does not depend on the device), fewer when that would
// be less than a step each.  A piece that lies
// within one share is stored to C; the parts of a piece cut by a share's
// boundary go to the workers' slots and f64_balanced_reduce_kernel adds them
// in order of k.
constexpr int kPiece = kF64Piece;
constexpr int kBalancedThreads = 256;

struct F64Spot {   // a place in the walk
  int64_t piece, step;
};

struct F64Balanced {
  const double* A;
  const double* B;
  double* C;
  double* slots;   // 2 per worker, kPiece x kPiece each
  F64Spot* starts;  // where each worker's share starts, then the end of the walk
  int64_t m, k, n;
  int64_t Mp, Np, Ks;   // pieces down and across, steps of 4 k
  int64_t rows16, cols8;  // live DMMA blocks: ceil(m / 16), ceil(n / 8)
  int workers;
  int64_t ranges;  // 0: a share may end after any step; s: only at the s-ths of k
};

// The start of worker i's share: at i / W of the DMMAs, rounded down to a step
// (to the start of its k range).
__device__ __forceinline__ F64Spot f64_spot(const F64Balanced& p, int i) {
  F64Spot s;
  if (i >= p.workers) {
    s.piece = p.Mp * p.Np;
    s.step = 0;
    return s;
  }
  const int64_t total = p.rows16 * p.cols8 * p.Ks;  // < 2^53
  const int64_t at = total / p.workers * i + total % p.workers * i / p.workers;
  const int64_t band = 2 * p.cols8 * p.Ks;          // a full row of pieces
  int64_t pm = at / band;
  if (pm > p.Mp - 1) pm = p.Mp - 1;
  int64_t rem = at - pm * band;
  const int64_t ml = p.rows16 - 2 * pm < 2 ? p.rows16 - 2 * pm : 2;
  int64_t pn = rem / (ml * 4 * p.Ks);
  if (pn > p.Np - 1) pn = p.Np - 1;
  rem -= pn * ml * 4 * p.Ks;
  const int64_t nl = p.cols8 - 4 * pn < 4 ? p.cols8 - 4 * pn : 4;
  s.piece = pm * p.Np + pn;
  s.step = rem / (ml * nl);
  if (p.ranges > 0) s.step = p.Ks * (s.step * p.ranges / p.Ks) / p.ranges;
  return s;
}

__global__ void __launch_bounds__(kBalancedThreads, 1) f64_balanced_kernel(
    const F64Balanced p, int* __restrict__ status) {
  release_next();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  // neighbouring shares on one sub-partition (warps w and w + 4)
  const int worker = blockIdx.x * (kBalancedThreads / 32) + (warp & 3) * 2 + (warp >> 2);
  if (worker >= p.workers) return;
  F64Spot at = f64_spot(p, worker);
  const F64Spot end = f64_spot(p, worker + 1);
  if (p.ranges != 1 && lane == 0) {
    p.starts[worker] = at;
    if (worker == p.workers - 1) p.starts[worker + 1] = end;
  }
  while (at.piece < end.piece || (at.piece == end.piece && at.step < end.step)) {
    const int64_t pm = at.piece / p.Np, pn = at.piece - pm * p.Np;
    const int64_t row0 = pm * kPiece, col0 = pn * kPiece;
    const int64_t s0 = at.step, s1 = at.piece < end.piece ? p.Ks : end.step;
    MXM_BOUNDS(row0 < p.m && col0 < p.n && s0 >= 0 && s1 <= p.Ks, status);
    const bool mlive1 = row0 + 16 < p.m;
    const int nlive = static_cast<int>(p.cols8 - 4 * pn < 4 ? p.cols8 - 4 * pn : 4);
    // this lane's A rows (halves g, g + 8 of the two m16 blocks) and B columns
    const double* ap[4];
    const double* bp[4];
    uint32_t rmask = 0, cmask = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t row = row0 + i * 8 + g, col = col0 + i * 8 + g;
      if (row < p.m) rmask |= 1u << i;
      if (col < p.n) cmask |= 1u << i;
      ap[i] = p.A + (row < p.m ? row : 0) * p.k + 4 * s0 + t4;
      bp[i] = p.B + (4 * s0 + t4) * p.n + (col < p.n ? col : 0);
    }
    int64_t kk = 4 * s0 + t4;  // this lane's k of the next load
    double acc[2][4][4];
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
      for (int ni = 0; ni < 4; ++ni)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[mi][ni][q] = 0.0;
    double a[4], b[4], an[4], bn[4];
    auto load = [&](double (&x)[4], double (&y)[4]) {
      const bool kv = kk < p.k;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        x[i] = (kv && ((rmask >> i) & 1u)) ? __ldg(ap[i]) : 0.0;
        y[i] = (kv && ((cmask >> i) & 1u)) ? __ldg(bp[i]) : 0.0;
        ap[i] += 4;
        bp[i] += 4 * p.n;
      }
      kk += 4;
    };
    load(a, b);
    f64_with_blocks(mlive1, nlive, [&](auto ml, auto nl) {
      for (int64_t s = s0; s < s1; ++s) {
        load(an, bn);
#pragma unroll
        for (int mi = 0; mi < decltype(ml)::value; ++mi)
#pragma unroll
          for (int ni = 0; ni < decltype(nl)::value; ++ni)
            dmma_16x8x4(acc[mi][ni], a[2 * mi], a[2 * mi + 1], b[ni]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          a[i] = an[i];
          b[i] = bn[i];
        }
      }
    });
    if (s0 == 0 && s1 == p.Ks) {
      // D fragment of m16n8: (g, 2 t4), (g, 2 t4 + 1), (g + 8, 2 t4), (g + 8, 2 t4 + 1)
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int64_t row = row0 + mi * 16 + h * 8 + g;
          if (row >= p.m) continue;
          double* crow = p.C + row * p.n;
#pragma unroll
          for (int ni = 0; ni < 4; ++ni) {
            const int64_t col = col0 + ni * 8 + 2 * t4;
            if (col < p.n) crow[col] = acc[mi][ni][2 * h];
            if (col + 1 < p.n) crow[col + 1] = acc[mi][ni][2 * h + 1];
          }
        }
      }
    } else {
      // slot 0: a piece begun by another worker, slot 1: one that this worker begins
      double* slot = p.slots + (static_cast<int64_t>(worker) * 2 + (s0 == 0 ? 1 : 0)) *
                                   (kPiece * kPiece) + lane;
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
#pragma unroll
          for (int q = 0; q < 4; ++q) slot[((mi * 4 + ni) * 4 + q) * 32] = acc[mi][ni][q];
    }
    ++at.piece;
    at.step = 0;
  }
}

// The pieces cut by share boundaries: block i takes the piece that worker i
// begins and does not finish (its elements shared over blockIdx.y) and adds
// the workers' parts in order of k.
__global__ void __launch_bounds__(kBalancedThreads) f64_balanced_reduce_kernel(
    const F64Balanced p) {
  follow_grid();
  const double* const slots = after_follow(p.slots);
  const int w0 = blockIdx.x;
  const F64Spot from = p.starts[w0], to = p.starts[w0 + 1];
  if (to.step == 0 || (from.piece == to.piece && from.step > 0)) return;
  const int64_t piece = to.piece;
  // the last worker that starts inside the piece
  int lo = w0 + 1, hi = p.workers - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.starts[mid].piece <= piece) lo = mid; else hi = mid - 1;
  }
  const int w1 = lo;
  const int64_t pm = piece / p.Np, pn = piece - pm * p.Np;
  for (int e = blockIdx.y * kBalancedThreads + threadIdx.x; e < kPiece * kPiece;
       e += gridDim.y * kBalancedThreads) {
    double v = slots[(static_cast<int64_t>(w0) * 2 + 1) * (kPiece * kPiece) + e];
    if (p.ranges == 0) {
#pragma unroll 8
      for (int w = w0 + 1; w <= w1; ++w)
        v += __ldcs(slots + static_cast<int64_t>(w) * 2 * (kPiece * kPiece) + e);
    } else {  // shares may be empty: those have no part
      for (int w = w0 + 1; w <= w1; ++w) {
        const F64Spot b = p.starts[w], n = p.starts[w + 1];
        if (b.piece < n.piece || b.step < n.step)
          v += __ldcs(slots + static_cast<int64_t>(w) * 2 * (kPiece * kPiece) + e);
      }
    }
    const int i = e >> 5, lane = e & 31, q = i & 3;
    const int64_t row = pm * kPiece + (i >> 4) * 16 + (q >> 1) * 8 + (lane >> 2);
    const int64_t col = pn * kPiece + ((i >> 2) & 3) * 8 + 2 * (lane & 3) + (q & 1);
    if (row < p.m && col < p.n) p.C[row * p.n + col] = v;
  }
}

}  // namespace

cudaError_t launch_f64_gemm(const double* A, const double* B, double* C, const F64Dims& d,
                            uint8_t* ws, size_t ws_bytes, int* status, cudaStream_t s) {
  if (d.m == 0 || d.n == 0 || d.k == 0) return cudaSuccess;
  F64Balanced p;
  p.A = A;
  p.B = B;
  p.C = C;
  p.slots = reinterpret_cast<double*>(ws);
  p.m = d.m;
  p.k = d.k;
  p.n = d.n;
  p.Mp = (d.m + kPiece - 1) / kPiece;
  p.Np = (d.n + kPiece - 1) / kPiece;
  p.Ks = (d.k + 3) / 4;
  p.rows16 = (d.m + 15) / 16;
  p.cols8 = (d.n + 7) / 8;
  p.ranges = d.ranges;
  int64_t workers = f64_workers(d);
  // a caller workspace of the packed copies' size may hold fewer slots
  const int64_t fit = static_cast<int64_t>(ws_bytes / kF64WorkerBytes) - 1;
  if (d.ranges != 1 && fit < workers) {
    if (fit < 64) p.ranges = 1;
    else workers = fit;
  }
  p.workers = static_cast<int>(workers);
  p.starts = reinterpret_cast<F64Spot*>(p.slots + workers * 2 * kPiece * kPiece);
  constexpr int kWarps = kBalancedThreads / 32;
  f64_balanced_kernel<<<(p.workers + kWarps - 1) / kWarps, kBalancedThreads, 0, s>>>(p, status);
  if (p.ranges != 1) {
    const unsigned split = p.Mp * p.Np < 304 ? kPiece * kPiece / kBalancedThreads : 1;
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e
                            : launch_chained(true, f64_balanced_reduce_kernel,
                                             dim3(p.workers, split), kBalancedThreads, 0, s, p);
  }
  return cudaGetLastError();
}

cudaError_t launch_f64_grouped(uint8_t* ws, int* status, cudaStream_t s) {
  // two resident CTAs of 8 warps per SM, every warp pulling pieces until the
  // cursor passes the last one
  f64_grouped_kernel<<<static_cast<unsigned>(2 * sm_count()), kGroupedF64Threads, 0, s>>>(ws,
                                                                                          status);
  return cudaGetLastError();
}

}  // namespace mxm
