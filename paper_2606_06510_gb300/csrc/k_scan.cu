// Phase 1 of Ozaki Scheme II (§2.3 Eq. scale; Algorithm 1 "scan the exponent
// spans of A, B; choose power-of-two diagonals D, E"): the exponent scan, the
// fallback flags, and the choice of D and E from the "+1" pass (§2.4).
#include <climits>

#include "k_scan.cuh"
#include "oz2_gemm.cuh"

namespace oz2 {

// Scan key of one element: 0 for zero, (frexp exponent + 2048) for a finite
// nonzero value (frexp exponent e: |x| = f·2^e, f ∈ [0.5, 1), so |x| < 2^e),
// and 1<<20 for Inf/NaN.  The max over a row is therefore the max-exponent
// of its finite entries, unless the row holds a non-finite value.
__device__ __forceinline__ int scan_key(double x) {
  unsigned long long b = __double_as_longlong(x);
  int E = static_cast<int>((b >> 52) & 0x7FF);
  unsigned long long mant = b & ((1ull << 52) - 1);
  if (E == 0x7FF) return 1 << 20;
  if (E == 0) {
    if (mant == 0) return 0;
    int bl = 64 - __clzll(static_cast<long long>(mant));  // bit length of the subnormal significand
    return bl - 1074 + 2048;
  }
  return E - 1022 + 2048;
}

// Rows of column-major A: thread per row, block row `by` of the k-chunks.
__device__ __forceinline__ void scan_a_rows(int64_t bx, int64_t by, int64_t m, int64_t k,
                                            const double* __restrict__ A, int64_t lda, int chunk,
                                            int* __restrict__ key) {
  int64_t i = bx * (int64_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  int64_t l0 = by * chunk;
  int64_t l1 = min(k, l0 + chunk);
  int best = 0;
  const double* p = A + i + l0 * lda;
  int64_t l = l0;
  for (; l + 8 <= l1; l += 8, p += 8 * lda) {  // eight loads in flight
    double x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = __ldg(p + j * lda);
#pragma unroll
    for (int j = 0; j < 8; ++j) best = max(best, scan_key(x[j]));
  }
  for (; l < l1; ++l, p += lda) best = max(best, scan_key(__ldg(p)));
  pdl_wait();  // the keys are zeroed (the operands were complete before that launch)
  if (best) atomicMax(key + i, best);
}

// Columns of column-major B: warp per column, lanes over l, block row `by`
// of the even-sized k-chunks; 16-byte loads when the column start is aligned.
__device__ __forceinline__ void scan_b_cols(int64_t bx, int64_t by, int64_t n, int64_t k,
                                            const double* __restrict__ B, int64_t ldb, int chunk, int vec,
                                            int* __restrict__ key) {
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t j = bx * (int64_t)(blockDim.x >> 5) + warp;
  if (j >= n) return;
  int64_t l0 = by * chunk;
  int64_t l1 = min(k, l0 + chunk);
  const double* col = B + j * ldb;
  int best = 0;
  if (vec) {
    const double2* c2 = reinterpret_cast<const double2*>(col);
    const int64_t p1 = l1 >> 1;  // pairs fully inside [l0, l1) (l0 is even)
    int64_t p = (l0 >> 1) + lane;
    for (; p < p1; p += 128) {  // four loads in flight, the last step's too
      double2 a[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) a[j] = p + 32 * j < p1 ? __ldg(c2 + p + 32 * j) : make_double2(0.0, 0.0);
#pragma unroll
      for (int j = 0; j < 4; ++j) best = max(best, max(scan_key(a[j].x), scan_key(a[j].y)));
    }
    if ((l1 & 1) && lane == 0) best = max(best, scan_key(__ldg(col + l1 - 1)));
  } else {
    int64_t l = l0 + lane;
    for (; l < l1; l += 128) {
      double a[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) a[j] = l + 32 * j < l1 ? __ldg(col + l + 32 * j) : 0.0;
#pragma unroll
      for (int j = 0; j < 4; ++j) best = max(best, scan_key(a[j]));
    }
  }
  best = __reduce_max_sync(0xffffffffu, best);
  pdl_wait();
  if (lane == 0 && best) atomicMax(key + j, best);
}

// Both operands in one launch: blocks [0, ga) scan rows of A (gax blocks of
// 256 rows per k-chunk), the rest scan columns of B (gbx blocks of 8 columns
// per k-chunk).
struct ScanGrid {
  int64_t ga, gax, gbx;
  int achunk, bchunk, vec;
};
__global__ void __launch_bounds__(256) scan_kernel(int64_t m, int64_t n, int64_t k, const double* __restrict__ A,
                                                   int64_t lda, const double* __restrict__ B, int64_t ldb, ScanGrid g,
                                                   int* __restrict__ ra, int* __restrict__ cb) {
  pdl_trigger();  // the flags kernel may be scheduled now; it waits for this grid to finish
  const int64_t b = blockIdx.x;
  if (b < g.ga) {
    scan_a_rows(b % g.gax, b / g.gax, m, k, A, lda, g.achunk, ra);
  } else {
    const int64_t bb = b - g.ga;
    scan_b_cols(bb % g.gbx, bb / g.gbx, n, k, B, ldb, g.bchunk, g.vec, cb);
  }
}

// One block per operand (block b takes operand first_op + b; 0: rows of A,
// 1: columns of B).  Decodes the scan keys, finds the lower median of the exponents of the nonzero finite rows,
// and writes the flags (bit0: native fallback; bit1: zero in the emulation)
// and the final exponent (0 for rows that are zero in the emulation).  With
// `lists` (two zeroed counts, then room for m rows and n columns) the flagged
// rows and columns are listed as well, which saves the fallback the launch
// that lists them (with its own launch as a dependent: 256³ 36.8 → 34.0 µs,
// 1000×777×1333 115.6 → 111.2, 2048³ at r = 8 255.3 → 251.8).
constexpr int kExpBins = 2112;   // frexp exponents of finite doubles: [-1073, 1024]
constexpr int kExpBias = 1080;
constexpr int kFinalizeThreads = 1024;
constexpr int kBinsPerThread = (kExpBins + kFinalizeThreads - 1) / kFinalizeThreads;

__global__ void __launch_bounds__(kFinalizeThreads) finalize_flags_kernel(int64_t m, int64_t n, int* __restrict__ ra,
                                      int* __restrict__ cb, uint8_t* __restrict__ row_flag,
                                      uint8_t* __restrict__ col_flag, unsigned flags,
                                      Oz2Device* dev, int first_op, int* __restrict__ lists) {
  __shared__ int hist[kExpBins];
  __shared__ int warp_sum[32];
  __shared__ int med_s;
  __shared__ int count_s;
  pdl_trigger();
  pdl_wait();  // the scan keys are complete
  const bool is_a = blockIdx.x + first_op == 0;
  const int64_t cnt = is_a ? m : n;
  int* key = is_a ? ra : cb;
  uint8_t* fl = is_a ? row_flag : col_flag;
  for (int b = threadIdx.x; b < kExpBins; b += blockDim.x) hist[b] = 0;
  if (threadIdx.x == 0) count_s = 0;
  __syncthreads();
  // Keys in batches of eight independent loads: one block reads them all, so
  // their latency is what this kernel takes for a large operand.
  constexpr int kBatch = 8;
  for (int64_t i0 = threadIdx.x; i0 < cnt; i0 += kBatch * kFinalizeThreads) {
    int kv[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) kv[j] = i0 + j * kFinalizeThreads < cnt ? key[i0 + j * kFinalizeThreads] : 0;
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
      if (kv[j] > 0 && kv[j] < (1 << 20)) atomicAdd(&hist[kv[j] - 2048 + kExpBias], 1);
  }
  __syncthreads();
  // Lower median of the histogram: each thread sums kBinsPerThread bins, a
  // block-wide inclusive scan of those sums locates the bin that holds the
  // element of rank ⌊(total-1)/2⌋.
  {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int b0 = threadIdx.x * kBinsPerThread;
    int mine = 0;
#pragma unroll
    for (int j = 0; j < kBinsPerThread; ++j) mine += b0 + j < kExpBins ? hist[b0 + j] : 0;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      int w = lane < kFinalizeThreads / 32 ? warp_sum[lane] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += v;
      }
      warp_sum[lane] = w;  // inclusive prefix over warps
    }
    __syncthreads();
    incl += wid ? warp_sum[wid - 1] : 0;
    const int total = warp_sum[kFinalizeThreads / 32 - 1];
    if (threadIdx.x == 0) med_s = 0;
    __syncthreads();
    if (total > 0) {
      const int rank = (total - 1) / 2;
      int acc = incl - mine;  // exclusive prefix
      if (acc <= rank && rank < incl) {
        for (int j = 0; j < kBinsPerThread; ++j) {
          acc += hist[b0 + j];
          if (acc > rank) {
            med_s = b0 + j - kExpBias;
            break;
          }
        }
      }
    }
    __syncthreads();
  }
  const int med = med_s;
  const bool window = (flags & OZ2_FLAG_NO_FALLBACK) == 0;
  int local = 0;
  for (int64_t i0 = threadIdx.x; i0 < cnt; i0 += kBatch * kFinalizeThreads) {
    int kv[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) kv[j] = i0 + j * kFinalizeThreads < cnt ? key[i0 + j * kFinalizeThreads] : 0;
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int64_t i = i0 + j * kFinalizeThreads;
      if (i >= cnt) break;
      const bool nonfinite = kv[j] >= (1 << 20);
      const bool nonzero = kv[j] > 0 && !nonfinite;
      const int e = nonzero ? kv[j] - 2048 : 0;
      const bool fb = nonfinite || (window && nonzero && abs(e - med) > kFallbackWindow);
      const bool zero = fb || !nonzero;
      fl[i] = static_cast<uint8_t>((fb ? 1 : 0) | (zero ? 2 : 0));
      key[i] = zero ? 0 : e;
      local += fb ? 1 : 0;
      if (fb && lists) lists[(is_a ? 2 : 2 + m) + atomicAdd(lists + (is_a ? 0 : 1), 1)] = static_cast<int>(i);
    }
  }
  if (local) atomicAdd(&count_s, local);
  __syncthreads();
  if (threadIdx.x == 0 && dev) {
    if (is_a) dev->fallback_rows = count_s;
    else dev->fallback_cols = count_s;
  }
}

cudaError_t launch_scan_keys(int64_t m, int64_t n, int64_t k, const double* A, int64_t lda, const double* B,
                             int64_t ldb, ScanOut out, cudaStream_t st, bool dependent) {
  if (k <= 0 || (m <= 0 && n <= 0)) return cudaSuccess;
  ScanGrid g{};
  // Rows of A: 64 k-entries per thread when that makes enough blocks to fill
  // the GPU (eight of 256 threads per SM), shorter runs down to 8 (one batch
  // of loads) when it does not: a small operand's scan is the latency of one
  // thread's run (256³: 64 entries 13.7 µs, 8 entries 3.2).
  g.gax = (m + 255) / 256;
  g.achunk = 64;
  while (g.achunk > 8 && g.gax * ((k + g.achunk - 1) / g.achunk) < 8 * num_sms()) g.achunk /= 2;
  int64_t ks = (k + g.achunk - 1) / g.achunk;
  if (ks > 65535) {
    g.achunk = static_cast<int>((k + 65534) / 65535);
    ks = (k + g.achunk - 1) / g.achunk;
  }
  // Columns of B: 1024 entries per warp, or one batch of loads (256) alike.
  g.gbx = (n + 7) / 8;
  g.bchunk = g.gbx * ((k + 1023) / 1024) < 8 * num_sms() ? 256 : 1024;
  int64_t bks = (k + g.bchunk - 1) / g.bchunk;
  if (bks > 65535) {
    g.bchunk = static_cast<int>((k + 65534) / 65535 + 1) & ~1;
    bks = (k + g.bchunk - 1) / g.bchunk;
  }
  g.ga = m > 0 ? g.gax * ks : 0;
  const int64_t gb = n > 0 ? g.gbx * bks : 0;
  g.vec = (ldb % 2 == 0) && (reinterpret_cast<uintptr_t>(B) % 16 == 0);
  if (g.ga + gb > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
  count_launch();
  // As a dependent of the kernel that zeroes the keys, the scan reads the
  // operands while that kernel runs; it must not where the operands are still
  // arriving, so the caller says (`dependent`).
  const dim3 grid(static_cast<unsigned>(g.ga + gb));
  if (dependent)
    return launch_dependent(scan_kernel, grid, dim3(256), 0, st, m, n, k, A, lda, B, ldb, g, out.ra, out.cb);
  scan_kernel<<<grid, 256, 0, st>>>(m, n, k, A, lda, B, ldb, g, out.ra, out.cb);
  return cudaGetLastError();
}

cudaError_t launch_scan_flags(int64_t m, int64_t n, int ops, unsigned flags, ScanOut out, Oz2Device* dev,
                              cudaStream_t st, int* lists) {
  if ((ops & 3) == 0) return cudaSuccess;
  const int first = (ops & 1) ? 0 : 1;
  const int count = ops == 3 ? 2 : 1;
  count_launch();
  const cudaError_t e = launch_dependent(finalize_flags_kernel, dim3(count), dim3(kFinalizeThreads), 0, st, m, n,
                                         out.ra, out.cb, out.row_flag, out.col_flag, flags, dev, first, lists);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_scan(int64_t m, int64_t n, int64_t k, const double* A, int64_t lda,
                        const double* B, int64_t ldb, unsigned flags, ScanOut out,
                        Oz2Device* dev, cudaStream_t st, bool zero_keys, int* lists) {
  cudaError_t err;
  // The scan keys are maxima taken with atomics: zero unless the caller has.
  if (zero_keys && m > 0 && (err = cudaMemsetAsync(out.ra, 0, sizeof(int) * m, st)) != cudaSuccess) return err;
  if (zero_keys && n > 0 && (err = cudaMemsetAsync(out.cb, 0, sizeof(int) * n, st)) != cudaSuccess) return err;
  if ((err = launch_scan_keys(m, n, k, A, lda, B, ldb, out, st, !zero_keys)) != cudaSuccess) return err;
  return launch_scan_flags(m, n, 3, flags, out, dev, st, lists);
}

// ---------------------------------------------------------------------------
// Scale choice (reading R-scale of the "+1" pass, or the crude bound R1).
// ---------------------------------------------------------------------------
// ⌈log2 U⌉ of a positive normal float.
__device__ __forceinline__ int ceil_log2_f32(float u) {
  unsigned b = __float_as_uint(u);
  int E = static_cast<int>((b >> 23) & 0xFF);
  return E - 127 + ((b & 0x7FFFFFu) ? 1 : 0);
}

__global__ void choose_scales_kernel(int64_t m, int64_t n, int64_t k, int T, int scale_mode,
                                     const float* __restrict__ urow, const int* u_max,
                                     const int* __restrict__ ra, const int* __restrict__ cb,
                                     const uint8_t* __restrict__ row_flag,
                                     const uint8_t* __restrict__ col_flag, int* __restrict__ d,
                                     int* __restrict__ e, Oz2Device* dev) {
  pdl_trigger();
  pdl_wait();
  int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int s, umax = 0;
  if (scale_mode == OZ2_SCALE_R2) {
    const int bits = *u_max;
    const float ug = __int_as_float(bits);
    if (idx == 0) dev->u_max_bits = bits;
    umax = ug > 0.f ? ceil_log2_f32(ug) : 0;
    s = min(62, (T - umax) >> 1);
  } else {
    int lk = k <= 1 ? 0 : 64 - __clzll(static_cast<long long>(k - 1));
    int pA = min(62, (T - lk) >> 1);
    s = min(62, T - lk - pA);
    if (idx < m) {
      d[idx] = (row_flag[idx] & 2) ? 0 : pA - ra[idx];
    } else if (idx < m + n) {
      int64_t j = idx - m;
      e[j] = (col_flag[j] & 2) ? 0 : s - cb[j];
    }
    if (idx == 0) dev->s = s;
    return;
  }
  if (idx < m) {
    float u = urow[idx];
    int ui = u > 0.f ? ceil_log2_f32(u) : umax;
    int t = min(62, T - s - ui);
    d[idx] = (row_flag[idx] & 2) ? 0 : t - ra[idx];
  } else if (idx < m + n) {
    int64_t j = idx - m;
    e[j] = (col_flag[j] & 2) ? 0 : s - cb[j];
  }
  if (idx == 0) dev->s = s;
}

cudaError_t launch_choose_scales(int64_t m, int64_t n, int64_t k, const Oz2Moduli& mods,
                                 int scale_mode, const float* urow, const int* u_max, const int32_t* ra,
                                 const int32_t* cb, const uint8_t* row_flag,
                                 const uint8_t* col_flag, int32_t* d, int32_t* e,
                                 Oz2Device* dev, cudaStream_t st) {
  int64_t tot = m + n;
  if (tot == 0) return cudaSuccess;
  count_launch();
  return launch_dependent(choose_scales_kernel, dim3(static_cast<unsigned>((tot + 255) / 256)), dim3(256), 0, st, m, n,
                          k, mods.T, scale_mode, urow, u_max, ra, cb, row_flag, col_flag, d, e, dev);
}

}  // namespace oz2
