// fft.cu -- the mod2f transform (Sec. 3.3): the 1-D complex DFT of Eq. 1,
// F(k) = sum_n f(n) W_N^{kn}, W_N = exp(-2 pi i / N), N a power of two,
// FP64 complex data interleaved (re, im).
//
// Eqs. 2-3 split a transform into radix-2 butterflies; the paper's
// split-stream form (tangle once, then every stage reads even / odd streams and
// concatenates up / down streams) is a layout for stream processors.  Here the
// stages of one sub-transform run in a CTA's shared memory, in the
// decimation-in-time order (input bit-reversed, output in place), and a
// transform too large for one CTA is cut in two passes over global memory (the
// "four-step" factorisation N = N1 N2, n = N2 n1 + n2, k = k1 + N1 k2):
//
//   pass 1: for every n2, the N1-point transform over n1 of x(N2 n1 + n2),
//           times the twiddle W_N^{n2 k1}, stored as Y[k1][n2];
//   pass 2: for every k1, the N2-point transform over n2 of Y[k1][.],
//           stored at X(k1 + N1 k2).
//
// FP64 is scarce on this GPU (a warp-wide FP64 instruction holds an SM
// sub-partition 64 clocks), so what counts is the number of FP64 instructions
// (the stages go two at a time, radix 4: 28 per 4 points and 2 stages, 16 in
// the twiddle-free first two) and that all sub-partitions have the same share
// of them: a CTA takes as many neighbouring columns as leave the waves of CTAs
// nearly full (2^20 points: one column, 1024 CTAs on 152 SMs; two columns, 512
// CTAs, fill 0.84 of theirs).  Indexes are shifts on 32 bits and signs flip by
// integers (a negation is an FP64 instruction: 39.5 + 33.5 a point before, 36 +
// 32 now).  Measured: 2^20 points 186 -> 158 us (the FP64 pipe alone 113 us, the
// rest the loads and stores at the ends of the passes and the barriers between
// stages; 6 us less since the second pass is launched beside the first), 2^10 11.2
// -> 8.7 us, 2^22 727 -> 665 us.  Butterflies of fused multiply-adds (a + w b in
// four, a - w b = 2 a - (a + w b) in two: 24 per radix 4) ran 2^20 points in
// 134 us, but with a tenth more error, and are not used.
#include <cuda_runtime.h>

#include <cstdint>

#include "mxm.h"
#include "mxm_internal.h"
#include "ptx.cuh"

namespace mxm {

int sm_count();

namespace {

constexpr int64_t kFftMaxN = int64_t{1} << 22;
constexpr int64_t kFftSingleMax = 1024;
constexpr int64_t kFftClusterMin = 16, kFftClusterMax = 8192;
constexpr int kFftClusterBits = 13;  // log2 of kFftClusterMax
// most dynamic shared memory of a CTA: of a pass (the rule of fft_column_bits),
// of a cluster (what a CTA may have beside its static part)
constexpr size_t kFftPassSmem = 96 * 1024, kFftClusterSmem = 200 * 1024;

// On this GPU a fused multiply-add of three registers issues every 64 clocks, an
// add, a multiply or a form with a constant operand every 76: sums and products
// go through fused multiply-adds with 1, -1 and -0 held in registers (read back
// from shared memory, so that the compiler does not know them; the results are
// those of the plain operations, signed zeros included).
struct Units {
  double one, mone, nzero;
};
__device__ __forceinline__ Units units() {
  __shared__ volatile double u[3];
  if (threadIdx.x == 0) {
    u[0] = 1.0;
    u[1] = -1.0;
    u[2] = -0.0;
  }
  __syncthreads();
  return Units{u[0], u[1], u[2]};
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b, const Units& k) {
  return make_double2(fma(a.x, k.one, b.x), fma(a.y, k.one, b.y));
}
__device__ __forceinline__ double2 csub(double2 a, double2 b, const Units& k) {
  return make_double2(fma(b.x, k.mone, a.x), fma(b.y, k.mone, a.y));
}
// a - i b and a + i b
__device__ __forceinline__ double2 csubi(double2 a, double2 b, const Units& k) {
  return make_double2(fma(b.y, k.one, a.x), fma(b.x, k.mone, a.y));
}
__device__ __forceinline__ double2 caddi(double2 a, double2 b, const Units& k) {
  return make_double2(fma(b.y, k.mone, a.x), fma(b.x, k.one, a.y));
}
// (a + bi)(c + di) with one rounding per component after a fused multiply-add
__device__ __forceinline__ double2 cmul(double2 a, double2 w, const Units& k) {
  return make_double2(fma(a.x, w.x, -fma(a.y, w.y, k.nzero)),
                      fma(a.x, w.y, fma(a.y, w.x, k.nzero)));
}

__device__ __forceinline__ uint32_t bitrev(uint32_t i, int bits) {
  return bits == 0 ? 0u : __brev(i) >> (32 - bits);
}

// W_T^j for 0 <= j < T from the half table (W_T^{j + T/2} = -W_T^j).
__device__ __forceinline__ double2 table_w(const double2* __restrict__ table, uint32_t T,
                                           uint32_t j) {
  const uint32_t h = T >> 1;
  if (j < h) return __ldg(table + j);
  const double2 w = __ldg(table + (j - h));
  // the sign bits by integers: a negation is an instruction of the FP64 pipe
  return make_double2(
      __hiloint2double(__double2hiint(w.x) ^ static_cast<int>(0x80000000u), __double2loint(w.x)),
      __hiloint2double(__double2hiint(w.y) ^ static_cast<int>(0x80000000u), __double2loint(w.y)));
}

// The decimation-in-time stages of C columns of L = 2^bits points in shared
// memory (data[c L + i], position i holding input bitrev(i); output in
// natural order), two at a time (radix 4): with h a quarter of the block,
// w = W_{4h}^j, j < h, and x_m at j + m h,
//   y0 = x0, y1 = w^2 x1, y2 = w x2, y3 = w^3 x3
//   x0, x2 = (y0 + y1) +- (y2 + y3);  x1, x3 = (y0 - y1) -+ i (y2 - y3)
// (the radix-2 stages of lengths 2h and 4h with W_{4h}^{j + h} = -i W_{4h}^j
// folded in).  An odd number of stages begins with the twiddle-free radix-2
// stage.  tw[m] = W_L^m, m < 3 L / 4.  All threads of the block call it; it
// ends with a barrier.
__device__ __forceinline__ void smem_fft(double2* data, const double2* tw, int bits, int C,
                                         const Units& k) {
  const int tid = threadIdx.x, nth = blockDim.x;
  const int L = 1 << bits;
  int hb = 0;  // h = 2^hb
  if (bits & 1) {
    for (int t = tid; t < C * (L >> 1); t += nth) {
      double2* p = data + 2 * t;
      const double2 x0 = p[0], x1 = p[1];
      p[0] = cadd(x0, x1, k);
      p[1] = csub(x0, x1, k);
    }
    __syncthreads();
    hb = 1;
  } else if (bits >= 2) {
    for (int t = tid; t < C * (L >> 2); t += nth) {
      double2* p = data + 4 * t;
      const double2 x0 = p[0], x1 = p[1], x2 = p[2], x3 = p[3];
      const double2 b0 = cadd(x0, x1, k), b1 = csub(x0, x1, k), b2 = cadd(x2, x3, k),
                    b3 = csub(x2, x3, k);
      p[0] = cadd(b0, b2, k);
      p[2] = csub(b0, b2, k);
      p[1] = csubi(b1, b3, k);
      p[3] = caddi(b1, b3, k);
    }
    __syncthreads();
    hb = 2;
  }
  for (; hb + 2 <= bits; hb += 2) {
    const int h = 1 << hb, ts = bits - hb - 2;  // W_{4h}^j = W_L^{j 2^ts}
    for (int t = tid; t < C * (L >> 2); t += nth) {
      const int j = t & (h - 1);
      double2* p = data + ((t - j) << 2) + j;  // columns follow each other: blocks of 4 h
      const int jt = j << ts;
      const double2 y0 = p[0], y1 = cmul(p[h], tw[2 * jt], k), y2 = cmul(p[2 * h], tw[jt], k),
                    y3 = cmul(p[3 * h], tw[3 * jt], k);
      const double2 b0 = cadd(y0, y1, k), b1 = csub(y0, y1, k), b2 = cadd(y2, y3, k),
                    b3 = csub(y2, y3, k);
      p[0] = cadd(b0, b2, k);
      p[2 * h] = csub(b0, b2, k);
      p[h] = csubi(b1, b3, k);
      p[3 * h] = caddi(b1, b3, k);
    }
    __syncthreads();
  }
}

struct FftPass {
  const double2* src;
  double2* dst;
  const double2* table;  // W_T^j, j < T/2
  int tbits;             // T = 2^tbits
  int bits1, bits2;      // N = N1 N2, N1 = 2^bits1; this pass transforms along N1 (stage 1) or N2
  int cbits;             // 2^cbits columns per CTA
  int stage;             // 1 or 2
};

// One CTA: C columns of an L-point transform in shared memory.
//   stage 1: column n2 = c0 + c reads x(N2 n1 + n2), n1 < L = N1; writes
//            Y[k1][n2] = Z(k1) W_N^{n2 k1} (with N2 = 1 this is the whole
//            transform, written in natural order, no twiddle);
//   stage 2: column k1 = c0 + c reads Y[k1][n2], n2 < L = N2; writes
//            X(k1 + N1 k2).
// Orders and columns are powers of two and N <= 2^22: shifts on 32 bits.
__global__ void __launch_bounds__(kFftThreads) fft_pass_kernel(const FftPass a) {
  extern __shared__ double2 sm[];
  const int C = 1 << a.cbits;
  const int bits = a.stage == 1 ? a.bits1 : a.bits2, L = 1 << bits;
  double2* data = sm;             // [C][L]
  double2* tw = sm + (C << bits); // W_L^m, m < 3 L / 4
  const int c0 = static_cast<int>(blockIdx.x) << a.cbits;
  const int tid = threadIdx.x, nth = blockDim.x;
  const Units k = units();

  // twiddles of the L-point transform: W_L^m = W_T^{m T / L}
  for (int m = tid; m < (3 * L + 3) / 4; m += nth)
    tw[m] = table_w(a.table, 1u << a.tbits, static_cast<uint32_t>(m) << (a.tbits - bits));
  // the second pass, launched beside the first, waits for its results here
  follow_grid();
  release_next();
  // load: C consecutive columns per row, c fastest
  for (int t = tid; t < (C << bits); t += nth) {
    const int r = t >> a.cbits, c = t & (C - 1), col = c0 + c;
    const int at = a.stage == 1 ? (r << a.bits2) + col : (col << a.bits2) + r;
    data[(c << bits) + bitrev(static_cast<uint32_t>(r), bits)] = a.src[at];
  }
  __syncthreads();

  smem_fft(data, tw, bits, C, k);

  const uint32_t nmask = (1u << (a.bits1 + a.bits2)) - 1u;
  for (int t = tid; t < (C << bits); t += nth) {
    const int kk = t >> a.cbits, c = t & (C - 1), col = c0 + c;
    double2 v = data[(c << bits) + kk];
    if (a.stage == 1) {
      if (a.bits2 > 0)
        v = cmul(v, table_w(a.table, 1u << a.tbits,
                            ((static_cast<uint32_t>(col) * static_cast<uint32_t>(kk)) & nmask)
                                << (a.tbits - a.bits1 - a.bits2)),
                 k);
      a.dst[(kk << a.bits2) + col] = v;  // Y[k1][n2]
    } else {
      a.dst[col + (kk << a.bits1)] = v;  // X(k1 + N1 k2)
    }
  }
}


// ---------------------------------------------------------------- one launch
// Transforms of up to kFftClusterMax points: both passes of the four-step
// factorisation in one launch of a thread-block cluster of C CTAs.  CTA r
// transforms the columns n2 in [r N2/C, (r + 1) N2/C) over n1, multiplies by
// W_N^{n2 k1} and writes each Y[k1][n2] straight into the shared memory of
// the CTA that owns row k1 in the second pass (rows [r N1/C, (r + 1) N1/C));
// after a cluster barrier every CTA transforms its rows over n2 and stores
// X(k1 + N1 k2).  The cluster barriers are hardware barriers; the only
// distributed-shared-memory writes come between the two, so no CTA can exit
// while a peer still writes to it.
struct FftCluster {
  const double2* src;
  double2* dst;
  const double2* table;
  int tbits, bits1, bits2;
};

__device__ __forceinline__ uint32_t fft_cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t fft_cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void fft_cluster_barrier() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\t"
      "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(kFftThreads) fft_cluster_kernel(const FftCluster a) {
  extern __shared__ double2 sm[];
  const int b1n = a.bits1, b2n = a.bits2, N1 = 1 << b1n, N2 = 1 << b2n;
  const int rank = static_cast<int>(fft_cluster_rank());
  const int sbits = 31 - __clz(static_cast<int>(fft_cluster_size()));
  const int cbits = b2n - sbits, rbits = b1n - sbits;  // columns of pass 1, rows of pass 2 per CTA
  double2* b1 = sm;                          // [cols][N1]
  double2* b2 = b1 + (N1 << cbits);          // [rows][N2], written by every CTA of the cluster
  double2* tw1 = b2 + (N2 << rbits);         // W_N1^m, m < 3 N1 / 4 (N1, N2 >= 4)
  double2* tw2 = tw1 + 3 * N1 / 4;           // W_N2^m, m < 3 N2 / 4
  const int tid = threadIdx.x;
  const Units k = units();
  const int c0 = rank << cbits, cols = 1 << cbits, rows = 1 << rbits;
  for (int t = tid; t < (N1 << cbits); t += kFftThreads) {
    const int r = t >> cbits, c = t & (cols - 1);
    b1[(c << b1n) + bitrev(static_cast<uint32_t>(r), b1n)] = a.src[(r << b2n) + c0 + c];
  }
  for (int m = tid; m < 3 * N1 / 4; m += kFftThreads)
    tw1[m] = table_w(a.table, 1u << a.tbits, static_cast<uint32_t>(m) << (a.tbits - b1n));
  for (int m = tid; m < 3 * N2 / 4; m += kFftThreads)
    tw2[m] = table_w(a.table, 1u << a.tbits, static_cast<uint32_t>(m) << (a.tbits - b2n));
  fft_cluster_barrier();  // every CTA runs (and has its tables) before any peer writes to it
  smem_fft(b1, tw1, b1n, cols, k);
  // Y[k1][n2] = Z_{n2}(k1) W_N^{n2 k1}, into row k1 % rows of CTA k1 / rows at
  // the place of n2 in the second transform's input order
  const uint32_t b2base = static_cast<uint32_t>(__cvta_generic_to_shared(b2));
  const uint32_t nmask = (1u << (b1n + b2n)) - 1u;
  for (int t = tid; t < (N1 << cbits); t += kFftThreads) {
    const int k1 = t >> cbits, c = t & (cols - 1), n2 = c0 + c;
    double2 v = b1[(c << b1n) + k1];
    v = cmul(v, table_w(a.table, 1u << a.tbits,
                        (static_cast<uint32_t>(n2 * k1) & nmask) << (a.tbits - b1n - b2n)),
             k);
    const uint32_t owner = static_cast<uint32_t>(k1 >> rbits);
    const uint32_t local =
        b2base + ((((k1 & (rows - 1)) << b2n) + bitrev(static_cast<uint32_t>(n2), b2n)) << 4);
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(owner));
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(remote), "d"(v.x), "d"(v.y)
                 : "memory");
  }
  fft_cluster_barrier();
  smem_fft(b2, tw2, b2n, rows, k);
  const int r0 = rank << rbits;
  for (int t = tid; t < (N2 << rbits); t += kFftThreads) {
    const int k2 = t >> rbits, c = t & (rows - 1);
    a.dst[r0 + c + (k2 << b1n)] = b2[(c << b2n) + k2];
  }
}

__global__ void fft_twiddle_kernel(double2* table, int64_t T) {
  const int64_t h = T >> 1;
  for (int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; j < h;
       j += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    double s, c;
    sincospi(static_cast<double>(j) / static_cast<double>(h), &s, &c);  // angle 2 pi j / T
    table[j] = make_double2(c, -s);
  }
}

bool pow2(int64_t v) { return v >= 1 && (v & (v - 1)) == 0; }

cudaError_t launch_pass(FftPass a, cudaStream_t s) {
  const int bits = a.stage == 1 ? a.bits1 : a.bits2;
  const int64_t cols = int64_t{1} << (a.stage == 1 ? a.bits2 : a.bits1);
  a.cbits = fft_column_bits(bits, cols, sm_count());
  const size_t L = size_t{1} << bits;
  const size_t smem = ((L << a.cbits) + (3 * L + 3) / 4) * sizeof(double2);
  static PerDevice limit;
  const cudaError_t e = allow_smem(limit, fft_pass_kernel, kFftPassSmem);
  if (e != cudaSuccess) return e;
  // a thread per radix-4 butterfly, up to 256
  int64_t threads = static_cast<int64_t>(L << a.cbits) / 4;
  threads = threads > kFftThreads ? kFftThreads : (threads < 32 ? 32 : threads);
  return launch_chained(a.stage == 2, fft_pass_kernel,
                        dim3(static_cast<unsigned>(cols >> a.cbits)),
                        dim3(static_cast<unsigned>(threads)), smem, s, a);
}

// One launch on a cluster of C CTAs (the largest power of two <= 16 that
// divides both factors), if the device can place it; cudaErrorNotSupported
// when it cannot, so that the caller takes the two-pass form.
cudaError_t launch_cluster(const FftCluster& a, cudaStream_t s) {
  static PerDevice limit, wide, fits[kFftClusterBits + 1];
  cudaError_t e = allow_smem(limit, fft_cluster_kernel, kFftClusterSmem);
  if (e != cudaSuccess) return e;
  int done = 0;
  e = wide.get(&done, [](int* v) {
    *v = 1;
    return cudaFuncSetAttribute(fft_cluster_kernel,
                                cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  });
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = {};
  auto configure = [&](int64_t C) {
    const size_t N1 = size_t{1} << a.bits1, N2 = size_t{1} << a.bits2;
    cfg.gridDim = dim3(static_cast<unsigned>(C), 1, 1);
    cfg.blockDim = dim3(kFftThreads, 1, 1);
    cfg.dynamicSmemBytes = (2 * (N1 * N2 / C) + 3 * (N1 + N2) / 4) * sizeof(double2);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(C);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  };
  // the cluster size that the device places, 0: none
  auto largest = [&](int* size) {
    int64_t C = 16;
    while (C > 1 && (C > (1 << a.bits1) || C > (1 << a.bits2))) C /= 2;
    for (*size = 0; C >= 1; C /= 2) {
      configure(C);
      int clusters = 0;
      const cudaError_t q = cudaOccupancyMaxActiveClusters(&clusters, fft_cluster_kernel, &cfg);
      if (q != cudaSuccess) return q;
      if (clusters >= 1) {
        *size = static_cast<int>(C);
        break;
      }
    }
    return cudaSuccess;
  };
  int size = 0;
  // bits1 - bits2 is 0 or 1, so their sum names the shape
  if ((e = fits[a.bits1 + a.bits2].get(&size, largest)) != cudaSuccess) return e;
  if (size == 0) return cudaErrorNotSupported;
  configure(size);
  e = cudaLaunchKernelEx(&cfg, fft_cluster_kernel, a);
  if (e == cudaSuccess) return e;
  // a context with fewer SMs than the one that was asked: ask for this one
  cudaGetLastError();
  if ((e = largest(&size)) != cudaSuccess) return e;
  return size == 0 ? cudaErrorNotSupported : cudaLaunchKernelEx(&cfg, fft_cluster_kernel, a);
}

}  // namespace

}  // namespace mxm

using namespace mxm;

extern "C" int64_t mxm_fft_max_n(void) { return kFftMaxN; }

extern "C" mxm_status mxm_fft_twiddles(double* table, int64_t n, void* stream) {
  NvtxRange nvtx_range("mxm_fft_twiddles");
  if (!pow2(n) || n > kFftMaxN) return MXM_ERR_INVALID_ARG;
  if (n < 2) return MXM_OK;  // no twiddle
  if (table == nullptr) return MXM_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(table) & 15) return MXM_ERR_ALIGNMENT;
  const int64_t h = n / 2;
  int64_t blocks = (h + 255) / 256;
  if (blocks > 4 * sm_count()) blocks = 4 * sm_count();
  fft_twiddle_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<double2*>(table), n);
  return cudaGetLastError() == cudaSuccess ? MXM_OK : MXM_ERR_CUDA;
}

extern "C" mxm_status mxm_fft(const double* in, double* out, double* work, const double* table,
                              int64_t table_n, int64_t n, void* stream) {
  NvtxRange nvtx_range("mxm_fft");
  if (!pow2(n) || n > kFftMaxN) return MXM_ERR_INVALID_ARG;
  if (in == nullptr || out == nullptr) return MXM_ERR_INVALID_ARG;
  if (n >= 2 && (table == nullptr || !pow2(table_n) || table_n < n || table_n > kFftMaxN))
    return MXM_ERR_INVALID_ARG;
  const bool two_pass = n > kFftSingleMax;
  if (two_pass && work == nullptr) return MXM_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out) |
       reinterpret_cast<uintptr_t>(work) | reinterpret_cast<uintptr_t>(table)) & 15)
    return MXM_ERR_ALIGNMENT;
  const size_t bytes = static_cast<size_t>(n) * 16;
  const auto overlap = [](const void* p, const void* q, size_t b) {
    const auto a0 = reinterpret_cast<uintptr_t>(p), b0 = reinterpret_cast<uintptr_t>(q);
    return a0 < b0 + b && b0 < a0 + b;
  };
  // out may be in (the passes read all of their source before the next
  // pass writes); work must be apart from both; a one-pass transform
  // reads and writes the same CTA's data but must not be in place across CTAs
  if (two_pass && (overlap(work, in, bytes) || overlap(work, out, bytes)))
    return MXM_ERR_INVALID_ARG;
  if (!two_pass && in != out && overlap(in, out, bytes)) return MXM_ERR_INVALID_ARG;
  const cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (n == 1) {
    return cudaMemcpyAsync(out, in, 16, cudaMemcpyDeviceToDevice, s) == cudaSuccess ? MXM_OK
                                                                                    : MXM_ERR_CUDA;
  }
  int p = 0, tp = 0;
  while ((int64_t{1} << p) < n) ++p;
  while ((int64_t{1} << tp) < table_n) ++tp;
  const int bits1 = (p + 1) / 2;
  cudaError_t e = cudaErrorNotSupported;
  if (n >= kFftClusterMin && n <= kFftClusterMax) {
    FftCluster c;
    c.src = reinterpret_cast<const double2*>(in);
    c.dst = reinterpret_cast<double2*>(out);
    c.table = reinterpret_cast<const double2*>(table);
    c.tbits = tp;
    c.bits1 = bits1;
    c.bits2 = p - bits1;
    e = launch_cluster(c, s);
    if (e == cudaSuccess) return MXM_OK;
    if (e != cudaErrorNotSupported) return MXM_ERR_CUDA;
  }
  FftPass a;
  a.table = reinterpret_cast<const double2*>(table);
  a.tbits = tp;
  a.cbits = 0;
  if (!two_pass) {
    a.src = reinterpret_cast<const double2*>(in);
    a.dst = reinterpret_cast<double2*>(out);
    a.bits1 = p;
    a.bits2 = 0;
    a.stage = 1;
    e = launch_pass(a, s);
  } else {
    a.bits1 = bits1;
    a.bits2 = p - bits1;
    a.src = reinterpret_cast<const double2*>(in);
    a.dst = reinterpret_cast<double2*>(work);
    a.stage = 1;
    e = launch_pass(a, s);
    if (e == cudaSuccess) {
      a.src = reinterpret_cast<const double2*>(work);
      a.dst = reinterpret_cast<double2*>(out);
      a.stage = 2;
      e = launch_pass(a, s);
    }
  }
  return e == cudaSuccess ? MXM_OK : MXM_ERR_CUDA;
}
