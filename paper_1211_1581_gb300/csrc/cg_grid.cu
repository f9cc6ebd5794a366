// cg_grid.cu -- conjugate gradients (Sec. 3.4) for systems too large for one
// thread-block cluster: the paper's `_while` loop runs inside one cooperative
// launch over all SMs, a block per SM, with three grid barriers a step:
//
//   product    q = A p on the block's own rows and its share of (p, q);
//   residual   (p, q) = the shares added in block order (the same sum in
//              every block); alpha = r2 / (p, q); r -= alpha q and the
//              block's share of (r, r);
//   direction  r2_new = the shares in block order; beta = r2_new / r2;
//              x += alpha p, p = r + beta p.
//
// Measured per step against three kernels in a conditional graph node (12 us
// of launches a step, every vector through memory): n = 10^6 with 7 diagonals
// 36.1 against 98.6 us (the FP64 pipe's share of it 19 us), 300,000 with 21
// 30.9 against 57.6, 12,288 with 511 25.7 against 46, 13,000 with 3 11.5
// against 16.2 (three barriers of 1.2 us, two dot products of 2 us each and
// the latency of one gather).
//
// Rows are shared out by number: block b of kCgBlocks owns rows
// [b n / kCgBlocks, (b + 1) n / kCgBlocks).  Where that gives a block more than
// twice the mean of the values, the rows are cut by work instead (cg_rows.h),
// once per solve: of 200,000 rows the first 1316 of 658 values, the rest of 3,
// 466 -> 101 us a step.  A block's q, r and x live in shared memory when they
// fit (n up to ~1.4 million; a block that the cut by work gives more rows than
// the mean keeps them in global memory), p, gathered by everybody, in global
// memory.  The product is bound by the FP64 pipe on this GPU (a warp-wide fused
// multiply-add holds an SM sub-partition 64 clocks, however many lanes are live)
// and by latency, so a row is given as few lanes as keep every thread on rows
// (one lane a row from 156,000 rows on: no shuffle tree, all 32 lanes live; the
// lanes' strided loads of values and columns meet in L1), and a lane has eight
// values, columns and gathers in flight.  Rows that are long beside the mean
// are taken by a whole warp, very long ones by the block (row_limit,
// block_limit): with those 1316 rows of 658 values 101 -> 29 us a step, a
// diagonal matrix of 160,001 rows bordered by one full row and column 16.5 ms ->
// 73 us, of 10^6 rows 103 ms -> 0.30 ms.
//
// The shares depend on the row pointers, the lanes per row on n and nnz only,
// and every sum has a fixed order: the rounding of a solve does not depend on the
// device (a device with room for fewer blocks gives each several).  Every
// wait at a barrier is bounded: after cg_wait_limit_ns it raises the abort word,
// records MXM_ERR_TIMEOUT and every block leaves.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "cg_rows.h"
#include "mxm.h"
#include "mxm_internal.h"

namespace mxm {

namespace {

constexpr int kCgGThreads = 1024;
constexpr int kCgGWarps = kCgGThreads / 32;
constexpr int64_t kCgGMaxShares = 1216;  // doubles per share table in the workspace
static_assert(3 * kCgBlocks <= kCgGMaxShares, "a share table, then the shares' rows");
constexpr int kBatch = 8;             // values, columns and gathers of a lane in flight

struct CgState {
  unsigned long long arrived;  // barrier arrivals since the start
  int abort;
};

struct CgWork {  // layout of the caller's workspace
  double* r;
  double* p;
  double* q;
  double* part_pq;
  double* part_rr;
  CgState* st;
};

size_t cg_workspace(int64_t n) {
  return static_cast<size_t>(3 * n + 2 * kCgGMaxShares + 4) * sizeof(double) + 256;
}

CgWork cg_work(double* w, int64_t n) {
  CgWork c;
  c.r = w;
  c.p = w + n;
  c.q = w + 2 * n;
  c.part_pq = w + 3 * n;
  c.part_rr = c.part_pq + kCgGMaxShares;
  c.st = reinterpret_cast<CgState*>(c.part_rr + kCgGMaxShares);
  return c;
}

struct CgGridArgs {
  const double* vals;
  const int32_t* indx;
  const int32_t* rowp;
  const double* b;
  double* x;
  CgWork w;
  int64_t n, nnz;
  int32_t row_limit, block_limit;  // longest row of the lanes, of a warp (cg_rows.h)
  int64_t rows_cap;   // most rows of a share by number
  int in_smem;        // q, r and x of a share of that many rows in shared memory
  double stop;
  uint64_t wait_ns;
  int32_t max_iters;
  int32_t* iters;
  double* r2;
  double* r2_hist;
  int* status;
};

// Sum of one double per thread in a fixed order; thread 0 gets it.  Four
// warps (one per sub-partition) add eight values each before their shuffle
// trees: every warp's own tree would hold the FP64 pipe four times as long.
__device__ __forceinline__ double block_total(double v, double* red) {
  const int tid = threadIdx.x;
  red[tid] = v;
  __syncthreads();
  if (tid < 128) {
    v = 0.0;
#pragma unroll
    for (int i = 0; i < kCgGThreads; i += 256) v += red[tid + i] + red[tid + i + 128];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if ((tid & 31) == 0) red[kCgGThreads + (tid >> 5)] = v;
  }
  __syncthreads();
  if (tid == 0)
    v = (red[kCgGThreads] + red[kCgGThreads + 1]) + (red[kCgGThreads + 2] + red[kCgGThreads + 3]);
  return v;
}

// The shares added in a fixed order by the first warp, and the step's
// quotient of the sum and r2 by one thread (an FP64 division by all of them
// would take a microsecond of the pipe): every thread gets both, the same in
// every block.
__device__ __forceinline__ void shares_total(const double* part, double* red, double r2,
                                             bool over, double& total, double& ratio) {
  double* const out = red + kCgGThreads + 4;
  if (threadIdx.x < 32) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < (kCgBlocks + 31) / 32; ++i) {
      const int s = i * 32 + threadIdx.x;
      const double v = s < kCgBlocks ? __ldcg(part + s) : 0.0;
      t = i == 0 ? v : t + v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    if (threadIdx.x == 0) {
      out[0] = t;
      out[1] = over ? r2 / t : t / r2;
    }
  }
  __syncthreads();
  total = out[0];
  ratio = out[1];
}

__device__ __forceinline__ uint64_t timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// All blocks; what each wrote before is visible to all after.  false: a wait
// gave up (here or in another block).
__device__ bool grid_barrier(CgState* st, unsigned long long& target, int* flag, uint64_t limit_ns,
                             int* status) {
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long seen;
    asm volatile("atom.add.release.gpu.global.u64 %0, [%1], 1;"
                 : "=l"(seen)
                 : "l"(&st->arrived)
                 : "memory");
    int ok = 1;
    const uint64_t t0 = timer_ns();
    for (uint32_t it = 1;; ++it) {
      asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(&st->arrived) : "memory");
      if (seen >= target) break;
      if ((it & 63u) == 0) {
        if (*reinterpret_cast<volatile int*>(&st->abort)) {
          ok = 0;
          break;
        }
        if (timer_ns() - t0 > limit_ns) {
          atomicExch(&st->abort, 1);
          atomicOr(status, kStatusTimeout);
          ok = 0;
          break;
        }
      }
    }
    *flag = ok;
  }
  __syncthreads();
  return *flag != 0;
}

// The pointers of a row (none: past the end, or the pointers are not in order);
// returns its length.
__device__ __forceinline__ int row_pointers(const CgGridArgs& a, int64_t row, int64_t hi, int& b,
                                            int& e) {
  b = e = 0;
  if (row < hi) {
    b = __ldg(a.rowp + row);
    e = __ldg(a.rowp + row + 1);
    if (b < 0 || e < b || e > a.nnz) b = e = 0;
  }
  return e - b;
}

// Thread `sub` of T's part of a row's sum.
template <int T>
__device__ __forceinline__ double cg_long_row(const CgGridArgs& a, int b, int e, int sub, bool& bad) {
  const double* const p = a.w.p;
  const int n = static_cast<int>(a.n);
  double t = 0.0;
  for (auto w = row_walk<int64_t>(b, e, sub); w.has(0); w.advance(kBatch * T)) {
    double v[kBatch], pv[kBatch];
    int c[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      c[u] = -1;
      v[u] = 0.0;
      if (w.has(u * T)) {
        c[u] = __ldg(a.indx + w.at + u * T);
        v[u] = __ldg(a.vals + w.at + u * T);
        bad |= c[u] < 0 || c[u] >= n;
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      pv[u] = 0.0;
      if (c[u] >= 0 && c[u] < n) pv[u] = __ldcg(p + c[u]);
      else v[u] = 0.0;
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) t = fma(v[u], pv[u], t);
  }
  return t;
}

// The rows of [lo, hi) that cg_product has left out: neighbours to different
// warps, then (huge) those for the whole block one after another.  Returns
// this thread's part of (p, q).  Out of line: its registers are its own.
struct LongRows {
  double pq;
  bool bad;
};
__device__ __noinline__ LongRows cg_long_rows(const CgGridArgs& a, int64_t lo, int64_t hi,
                                              double* qs, bool huge, double* red) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* const p = a.w.p;
  double pq = 0.0;
  bool bad = false;
  int b, e;
  for (int64_t base = lo; base < hi; base += kCgGThreads) {
    const int len = row_pointers(a, base + lane * kCgGWarps + warp, hi, b, e);
    for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, len > a.row_limit && len <= a.block_limit);
         todo != 0; todo &= todo - 1) {
      const int src = __ffs(todo) - 1;
      double t = cg_long_row<32>(a, __shfl_sync(0xFFFFFFFFu, b, src),
                                 __shfl_sync(0xFFFFFFFFu, e, src), lane, bad);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
      if (lane == 0) {
        const int64_t row = base + src * kCgGWarps + warp;
        qs[row - lo] = t;
        pq = fma(__ldcg(p + row), t, pq);
      }
    }
  }
  if (!huge) return LongRows{pq, bad};  // block-uniform
  for (int64_t base = lo; base < hi; base += kCgGThreads) {
    if (!__syncthreads_or(row_pointers(a, base + tid, hi, b, e) > a.block_limit)) continue;
    for (int64_t base32 = base; base32 < base + kCgGThreads; base32 += 32) {  // all warps alike
      const int len = row_pointers(a, base32 + lane, hi, b, e);
      for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, len > a.block_limit); todo != 0;
           todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        const double t =
            block_total(cg_long_row<kCgGThreads>(a, __shfl_sync(0xFFFFFFFFu, b, src),
                                                 __shfl_sync(0xFFFFFFFFu, e, src), tid, bad), red);
        if (tid == 0) {
          qs[base32 + src - lo] = t;
          pq = fma(__ldcg(p + base32 + src), t, pq);
        }
      }
    }
  }
  return LongRows{pq, bad};
}

// q = A p on rows [lo, hi) (qs[row - lo]); returns this thread's part of
// (p, q).  G lanes a row; a warp takes 32 / G rows at a time.  kUneven: rows
// longer than row_limit are left out; any number of values, else kNarrowValues.
template <int G, bool kUneven>
__device__ __forceinline__ double cg_product(const CgGridArgs& a, int64_t lo, int64_t hi,
                                             double* qs, bool& bad) {
  constexpr int R = 32 / G;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = lane & (G - 1), grp = lane / G;
  const double* const p = a.w.p;
  const int n = static_cast<int>(a.n);
  double pq = 0.0;
  for (int64_t base = lo + static_cast<int64_t>(warp) * R; base < hi;
       base += static_cast<int64_t>(kCgGWarps) * R) {
    const int64_t row = base + grp;
    int b = 0, e = 0;
    double prow = 0.0;
    bool own = row < hi;
    if (own) {
      b = __ldg(a.rowp + row);
      e = __ldg(a.rowp + row + 1);
      if (b < 0 || e < b || e > a.nnz) {
        bad = true;
        b = e = 0;
      }
      if (kUneven && e - b > a.row_limit) {
        own = false;
        b = e = 0;
      }
      if (sub == 0) prow = __ldcg(p + row);
    }
    auto w = row_walk<std::conditional_t<kUneven, int64_t, int32_t>>(b, e, sub);
    double t = 0.0;
    // the most values any lane of the warp has left (the warp runs together)
    int m = __reduce_max_sync(0xFFFFFFFFu, w.count(G));
    for (; m > 0; m -= kBatch) {
      double v[kBatch], pv[kBatch];
      int c[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        c[u] = -1;
        v[u] = 0.0;
        if (w.has(u * G)) {
          c[u] = __ldg(a.indx + w.at + u * G);
          v[u] = __ldg(a.vals + w.at + u * G);
          bad |= c[u] < 0 || c[u] >= n;
        }
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        pv[u] = 0.0;
        if (c[u] >= 0 && c[u] < n) pv[u] = __ldcg(p + c[u]);
        else v[u] = 0.0;
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        if (u < m) t = fma(v[u], pv[u], t);  // uniform
      w.advance(kBatch * G);
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    if (own && sub == 0) {
      qs[row - lo] = t;
      pq = fma(prow, t, pq);
    }
  }
  return pq;
}

// A solve.  kUneven: the shares' rows as this block has left them in `span`, rows
// beyond row_limit done apart, positions in 64 bits; compiled apart, since the
// way to the rows alone costs 1.5 us a step.  Both meet at the same barriers.
template <int G, bool kUneven>
__device__ __forceinline__ void cg_solve(const CgGridArgs& a, double* dsm, double* red, int& flag,
                                         const int64_t* span, bool any_long, bool any_huge) {
  const int tid = threadIdx.x;
  const bool many = gridDim.x < kCgBlocks;  // several shares a block: their vectors in memory
  CgState* const st = a.w.st;
  unsigned long long target = 0;
  bool bad = false;
  auto lo_of = [&](int s) { return kUneven ? __ldcg(span + 2 * s) : share_by_rows(a.n, s); };
  auto hi_of = [&](int s) { return kUneven ? __ldcg(span + 2 * s + 1) : share_by_rows(a.n, s + 1); };
  const bool smem = a.in_smem && !many &&
                    (!kUneven || hi_of(blockIdx.x) - lo_of(blockIdx.x) <= a.rows_cap);
  auto q_of = [&](int64_t lo) { return smem ? dsm : a.w.q + lo; };
  auto r_of = [&](int64_t lo) { return smem ? dsm + a.rows_cap : a.w.r + lo; };
  auto x_of = [&](int64_t lo) { return smem ? dsm + 2 * a.rows_cap : a.x + lo; };

  // x0 = 0, r0 = p0 = b, shares of (b, b)
  for (int s = blockIdx.x; s < kCgBlocks; s += gridDim.x) {
    const int64_t lo = lo_of(s), hi = hi_of(s);
    double* const r = r_of(lo);
    double* const x = x_of(lo);
    double bb = 0.0;
    for (int64_t i = lo + tid; i < hi; i += kCgGThreads) {
      const double bi = __ldg(a.b + i);
      x[i - lo] = 0.0;
      r[i - lo] = bi;
      a.w.p[i] = bi;
      bb = fma(bi, bi, bb);
    }
    bb = block_total(bb, red);
    if (tid == 0) a.w.part_rr[s] = bb;
  }
  bool ok = grid_barrier(st, target, &flag, a.wait_ns, a.status);
  double r2 = 0.0, unused;
  if (ok) shares_total(a.w.part_rr, red, 1.0, false, r2, unused);
  int32_t k = 0;
  bool brk = false;
  while (ok && r2 > a.stop && k < a.max_iters) {
    for (int s = blockIdx.x; s < kCgBlocks; s += gridDim.x) {
      const int64_t lo = lo_of(s), hi = hi_of(s);
      double pq = cg_product<G, kUneven>(a, lo, hi, q_of(lo), bad);
      if (kUneven && any_long) {
        const LongRows rest = cg_long_rows(a, lo, hi, q_of(lo), any_huge, red);
        pq += rest.pq;
        bad |= rest.bad;
      }
      pq = block_total(pq, red);
      if (tid == 0) a.w.part_pq[s] = pq;
    }
    if (!(ok = grid_barrier(st, target, &flag, a.wait_ns, a.status))) break;
    double pAp, alpha, r2n, beta;
    shares_total(a.w.part_pq, red, r2, true, pAp, alpha);
    if (!(pAp > 0.0)) {  // the same in every block: the same shares, the same order
      brk = true;
      break;
    }
    for (int s = blockIdx.x; s < kCgBlocks; s += gridDim.x) {
      const int64_t lo = lo_of(s), own = hi_of(s) - lo;
      const double* const q = q_of(lo);
      double* const r = r_of(lo);
      double rr = 0.0;
      for (int64_t i = tid; i < own; i += kCgGThreads) {
        const double ri = fma(-alpha, q[i], r[i]);
        r[i] = ri;
        rr = fma(ri, ri, rr);
      }
      rr = block_total(rr, red);
      if (tid == 0) a.w.part_rr[s] = rr;
    }
    if (!(ok = grid_barrier(st, target, &flag, a.wait_ns, a.status))) break;
    shares_total(a.w.part_rr, red, r2, false, r2n, beta);
    r2 = r2n;
    for (int s = blockIdx.x; s < kCgBlocks; s += gridDim.x) {
      const int64_t lo = lo_of(s), own = hi_of(s) - lo;
      const double* const r = r_of(lo);
      double* const x = x_of(lo);
#pragma unroll 4
      for (int64_t i = tid; i < own; i += kCgGThreads) {
        const double pi = __ldcg(a.w.p + lo + i);
        x[i] = fma(alpha, pi, x[i]);
        __stcg(a.w.p + lo + i, fma(beta, pi, r[i]));
      }
    }
    if (blockIdx.x == 0 && tid == 0 && a.r2_hist != nullptr) a.r2_hist[k] = r2;
    ++k;
    if (!(ok = grid_barrier(st, target, &flag, a.wait_ns, a.status))) break;
  }
  if (smem) {  // each thread's own elements
    const int64_t lo = lo_of(blockIdx.x), own = hi_of(blockIdx.x) - lo;
    for (int64_t i = tid; i < own; i += kCgGThreads) a.x[lo + i] = x_of(lo)[i];
  }
  if (blockIdx.x == 0 && tid == 0) {
    *a.iters = k;
    *a.r2 = r2;
    if (brk) atomicOr(a.status, kStatusBreakdown);
  }
  if (bad) atomicOr(a.status, kStatusBounds);
}

template <int G>
__global__ void __launch_bounds__(kCgGThreads, 1) cg_grid_kernel(const __grid_constant__ CgGridArgs a) {
  extern __shared__ double dsm[];
  __shared__ double red[kCgGThreads + 6];
  __shared__ int flag;
  const int tid = threadIdx.x;
  // The shares' rows: by number, or (the same choice in every block) by work,
  // each block then looking its own up and keeping them behind the share table.
  int64_t* const span = reinterpret_cast<int64_t*>(a.w.part_pq + kCgBlocks);
  bool too_long = false;
  if (tid < kCgBlocks) {
    const int64_t first = __ldg(a.rowp + share_by_rows(a.n, tid));
    too_long = share_too_long(__ldg(a.rowp + share_by_rows(a.n, tid + 1)) - first, a.nnz);
  }
  const bool by_work = __syncthreads_or(too_long) != 0;
  int longest = 0;  // of the block's rows, by this thread
  for (int s = blockIdx.x; s < kCgBlocks; s += gridDim.x) {
    int64_t lo = share_by_rows(a.n, s), hi = share_by_rows(a.n, s + 1);
    if (by_work) {
      if (tid < 2) span[2 * s + tid] = share_by_work(a.rowp, a.n, a.nnz, s + tid);
      __syncthreads();
      lo = __ldcg(span + 2 * s);
      hi = __ldcg(span + 2 * s + 1);
    }
    for (int64_t i = lo + tid; i < hi; i += kCgGThreads) {
      int b, e;
      longest = max(longest, row_pointers(a, i, hi, b, e));
    }
  }
  const bool any_long = __syncthreads_or(longest > a.row_limit) != 0;
  if (!by_work && !any_long && a.nnz <= kNarrowValues) {
    cg_solve<G, false>(a, dsm, red, flag, nullptr, false, false);
    return;
  }
  if (!by_work)
    for (int s = blockIdx.x; s < kCgBlocks; s += gridDim.x)
      if (tid < 2) span[2 * s + tid] = share_by_rows(a.n, s + tid);
  // (a barrier of the block: the span is read after it)
  const bool any_huge = __syncthreads_or(longest > a.block_limit) != 0;
  cg_solve<G, true>(a, dsm, red, flag, span, any_long, any_huge);
}

// Lanes per row: the fewest that give every thread of a share a row.
int cg_grid_group(int64_t n, int64_t nnz) {
  const int64_t rows = (n + kCgBlocks - 1) / kCgBlocks;
  const int64_t avg = n > 0 ? (nnz + n - 1) / n : 0;
  int g = 1;
  while (g < 32 && rows * g < kCgGThreads && g < avg) g *= 2;
  return g;
}

// The most dynamic shared memory of a block and the most blocks at once are asked
// of the device once, and the limit raised once: solves of different orders from
// two threads would lower it under each other between a call and its launch.
template <int G>
mxm_status launch_grid(CgGridArgs a, cudaStream_t s) {
  static PerDevice limit, held;
  int most = 0, blocks = 0;
  const cudaError_t e = limit.get(&most, [](int* v) {
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t q = cudaGetDevice(&dev);
    if (q == cudaSuccess)
      q = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (q == cudaSuccess) q = cudaFuncGetAttributes(&fa, cg_grid_kernel<G>);
    if (q != cudaSuccess) return q;
    *v = optin - static_cast<int>(fa.sharedSizeBytes);
    return cudaFuncSetAttribute(cg_grid_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, *v);
  });
  if (e != cudaSuccess) return MXM_ERR_CUDA;
  if (held.get(&blocks, [&](int* v) {  // a block fills an SM's registers, whatever its memory
        int dev = 0, sms = 0, per_sm = 0;
        cudaError_t q = cudaGetDevice(&dev);
        if (q == cudaSuccess) q = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (q == cudaSuccess)
          q = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cg_grid_kernel<G>, kCgGThreads,
                                                            static_cast<size_t>(most));
        *v = sms * per_sm;
        return q;
      }) != cudaSuccess)
    return MXM_ERR_CUDA;
  a.row_limit = row_limit(a.n, a.nnz, G);
  a.block_limit = block_limit(a.row_limit);
  a.rows_cap = (a.n + kCgBlocks - 1) / kCgBlocks;
  size_t smem = 3 * static_cast<size_t>(a.rows_cap) * sizeof(double);
  a.in_smem = smem <= static_cast<size_t>(most) ? 1 : 0;
  if (!a.in_smem) smem = 0;
  if (blocks > kCgBlocks) blocks = kCgBlocks;
  if (blocks < 1) return MXM_ERR_CUDA;
  if (cudaMemsetAsync(a.w.st, 0, sizeof(CgState), s) != cudaSuccess) return MXM_ERR_CUDA;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(reinterpret_cast<void*>(cg_grid_kernel<G>), dim3(blocks),
                                     dim3(kCgGThreads), args, smem, s) == cudaSuccess
             ? MXM_OK
             : MXM_ERR_CUDA;
}

}  // namespace

size_t cg_grid_workspace_bytes(int64_t n) { return cg_workspace(n); }

// One solve by the engine over all SMs (arguments checked by the caller).
mxm_status cg_grid_solve(const double* vals, const int32_t* indx, const int32_t* rowp,
                         const double* b, double* x, double* work, int32_t* iters, double* r2,
                         double* r2_hist, int64_t n, int64_t nnz, double stop,
                         int32_t max_iters, int* status, cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) return MXM_ERR_CUDA;
  if (cap != cudaStreamCaptureStatusNone) return MXM_ERR_UNSUPPORTED;
  CgGridArgs a;
  a.vals = vals;
  a.indx = indx;
  a.rowp = rowp;
  a.b = b;
  a.x = x;
  a.w = cg_work(work, n);
  a.n = n;
  a.nnz = nnz;
  a.row_limit = a.block_limit = 0;
  a.rows_cap = 0;
  a.in_smem = 0;
  a.stop = stop;
  a.wait_ns = cg_wait_limit_ns(nnz);
  a.max_iters = max_iters;
  a.iters = iters;
  a.r2 = r2;
  a.r2_hist = r2_hist;
  a.status = status;
  switch (cg_grid_group(n, nnz)) {
    case 1: return launch_grid<1>(a, s);
    case 2: return launch_grid<2>(a, s);
    case 4: return launch_grid<4>(a, s);
    case 8: return launch_grid<8>(a, s);
    case 16: return launch_grid<16>(a, s);
    default: return launch_grid<32>(a, s);
  }
}

}  // namespace mxm
