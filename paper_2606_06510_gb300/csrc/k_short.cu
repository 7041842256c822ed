// C for a short k (k ≤ 64) without residues: the product ÃB̃ of the scaled
// integer matrices (Algorithm 1 "lin:quant") from their base-256 digits.
//
// Per output the residue path costs r accumulator pairs drained and reduced,
// 2r bytes written and read back, and a CRT sum, whatever k is; with one
// k-block per unit that is all it does (16384²×64, r = 12: 2.39 ms of residue
// GEMM and 2.05 ms of reconstruction for 0.26 ms of plane products).  For a
// short k the integer X_ij = Σ_l Ã_il B̃_lj itself can be formed on the tensor
// cores: with balanced digits Ã = Σ_i a_i 256^i, a_i ∈ [-128, 127] (at most 8:
// |Ã| < 2^62), the digit products of equal weight share an accumulator,
//   acc_w = Σ_{i+j=w} Σ_l a_i b_j,  |acc_w| ≤ 8·64·2^14 = 2^23,
// exact in FP32 (f16 operands, kind::f16), and X = Σ_w acc_w 256^w, at most
// 15 terms.  The scales bound |X| by 2^T < M/2, so X is the integer the CRT
// would return, and the same rounding gives the same bits of C.
//
// A CTA works on 128 rows × 16 columns of C at a time.  Operand B's tile
// stacks the 16 columns of digit 0, then of digit 1, and so on, with zero
// lines before and after: an MMA of digit i of A with the tile shifted by i
// mod 4 digits adds the products a_i·b_j of every j to the 16 columns of
// weight i + j, so that four digits of A share one accumulator window (moving
// the window stalls the tensor core) and a tile has two windows.  240 of 256
// columns are used, and two such buffers let the epilogue work on one tile
// while the tensor core fills the other.  The A digits of a row block (8 tiles
// of 16 KiB at most) stay in shared memory while the CTA walks along its
// columns; that is what limits k to 64 (the sums stay exact up to 128).
//
// Flagged rows, when they are few, are recomputed meanwhile by two more warps
// of every CTA, on the FP64 pipe that nothing else here uses.
//
// Measured on one GB300, 16384²×64, r = 12 (268 M outputs): 2.0 ms for this
// kernel, where the residue GEMM and the reconstruction took 2.47 + 2.02 ms
// (the call 4.70 → 2.15 ms; k = 32 4.69 → 1.75, k = 16 4.69 → 1.66; r = 6
// 3.14 → 1.54).  The MMAs alone take 1.45 ms (88 cycles each, the rate of
// M = 128, N = 176 f16), the epilogue alone somewhat more (some 130
// instructions per output); together the tensor pipe is about 60% active, its
// issue slowed by the epilogue warps.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "oz2_crt.cuh"
#include "oz2_gemm.cuh"
#include "oz2_quant.cuh"

namespace oz2 {

constexpr int kSkDigits = 8;                       // base-256 digits of an integer below 2^62
constexpr int kSkK = 64;                           // k-entries of an operand line (128 bytes of f16)
constexpr int kSkCols = 16;                        // columns of C per tile
constexpr int kSkClasses = 2 * kSkDigits - 1;      // weights i + j
constexpr int kSkStages = 3;                       // B tiles in flight
constexpr int kSkGroup = 4;                        // digits of A that share an accumulator window
constexpr int kSkPad = (kSkGroup - 1) * kSkCols * kPlaneLine;  // zero lines on both sides of a B tile
constexpr int kSkStageStep = kTileBytes + kSkPad;  // the pad after one tile is the one before the next
constexpr int kSkBufCols = 256;                    // TMEM columns of an accumulator buffer
constexpr int kSkEpiWarps = 16;
constexpr int kSkNativeWarps = 2, kSkNativeRows = 4;
constexpr int kSkThreads = 32 * (2 + kSkEpiWarps + kSkNativeWarps);  // producer, MMA issuer, epilogue, native FP64
constexpr int kSkDigitThreads = 1024;              // 128 rows × 8 threads of 8 entries
static_assert(kSkClasses * kSkCols <= kSkBufCols && 2 * kSkBufCols <= 512, "two buffers in tensor memory");
static_assert(kSkDigits * kSkCols == kRows, "a B tile is one 128-line block");

struct ShortArgs {
  int64_t m, n, nrb, nct, ldc, nbb;  // row blocks of A, column tiles of B, 128-column blocks of B
  int ksteps;                        // MMA K-steps (16 entries)
  const int *na, *nb;                // digits of each row block of A, of each 128 columns of B
  const int *d, *e;
  double* C;
  Oz2Device* dev;
  NativeRows fb;
  int64_t k;
  int pow256[4];  // 1, 256, 256², 256³: as data, so that the sums stay multiply-adds (as
                  // constants they become shifts and adds, four instructions for one)
};

// ---------------------------------------------------------------------------
// The digits, as f16, in the operand tiles: line (row block·8 + digit)·128 +
// row of A, line column tile·128 + 16·digit + column of B, 64 k-entries each
// (zero past k, past the operand's rows and in rows the flags zero).  A block
// takes 128 rows and records how many digits they need.
// ---------------------------------------------------------------------------
struct DigitOperand {
  const double* base;
  int64_t row_stride, k_stride, rows, lines_rows;  // lines_rows: rows stored (A: to 128, B: to 16)
  const int *exps, *scan;                          // d or e, and ra or cb
  const uint8_t* flag;
  uint8_t* out;
  int* digits;
};

__global__ void __launch_bounds__(kSkDigitThreads) short_digits_kernel(DigitOperand X0, DigitOperand X1, int blocks0,
                                                                       int k) {
  pdl_trigger();
  pdl_wait();
  __shared__ int need_s;
  const bool is_b = static_cast<int>(blockIdx.x) >= blocks0;
  const DigitOperand X = is_b ? X1 : X0;
  const int64_t blk = is_b ? blockIdx.x - blocks0 : blockIdx.x;
  const int rloc = threadIdx.x >> 3, part = threadIdx.x & 7;
  const int64_t row = blk * kRows + rloc;
  if (threadIdx.x == 0) need_s = 1;
  __syncthreads();
  unsigned long long u[8];  // Ã + 128·(256^8 - 1)/255: its bytes are the balanced digits plus 128
#pragma unroll
  for (int j = 0; j < 8; ++j) u[j] = 0x8080808080808080ull;
  if (row < X.rows && !(X.flag[row] & 2)) {
    const int d = X.exps[row];
    const double* p = X.base + row * X.row_stride + part * 8 * X.k_stride;
    double x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = part * 8 + j < k ? __ldg(p + j * X.k_stride) : 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) u[j] += quantise_entry(x[j], d, false);
    // |Ã| ≤ 2^t with t = d + (max-exponent): n digits hold ±2^(8n - 2).
    if (part == 0) atomicMax(&need_s, min(kSkDigits, (d + X.scan[row] + 9) >> 3));
  }
  if (row < X.lines_rows) {
    const int64_t line = is_b ? (row / kSkCols) * kRows + row % kSkCols : blk * kSkDigits * kRows + rloc;
    uint8_t* dst = X.out + line * kPlaneLine + part * 16;
    const int64_t step = static_cast<int64_t>(is_b ? kSkCols : kRows) * kPlaneLine;
#pragma unroll
    for (int i = 0; i < kSkDigits; ++i) {
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t a = static_cast<uint32_t>(u[2 * j] >> (32 * (i >> 2))), b = static_cast<uint32_t>(u[2 * j + 1] >> (32 * (i >> 2)));
        // Bytes i of both as halves 1024 + byte, then less 1152.
        const uint32_t two = __byte_perm(a, b, (i & 3) | ((4 + (i & 3)) << 4));
        const uint32_t h = __byte_perm(two, 0x64646464u, 0x4140);
        const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(0x6480)));
        w[j] = *reinterpret_cast<const uint32_t*>(&v);
      }
      *reinterpret_cast<uint4*>(dst + i * step) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) X.digits[blk] = need_s;
}

// ---------------------------------------------------------------------------
// Digit products and C.
// ---------------------------------------------------------------------------
// The digit counts a launch runs with, for operands that need na and nb:
// digits that are all zero make the weights, na + nb - 1, a multiple of four
// (or all 15), since the epilogue takes them in fours.  They go to B first: a
// digit of A is products of its own, one of B only widens them (8192²×64, A
// first and B first: r = 4 439 and 327 µs a call, r = 6 413 and 351, r = 8 557
// and 490, r ≥ 10 alike).
struct DigitCounts {
  int a, b;
};
__device__ __forceinline__ DigitCounts digit_counts(int na, int nb) {
  const int more = (1 - na - nb) & 3;
  const int b = min(kSkDigits, nb + more);
  return {min(kSkDigits, na + nb + more - b), b};
}

// Flagged rows by FP64 FMA chains in the order of k, as fma_gemm_kernel forms
// them: a warp takes kSkNativeRows rows × 32 columns, a lane a column, the rows'
// entries in shared memory.
__device__ __forceinline__ void native_rows(const ShortArgs& a, int nr, int worker, int workers,
                                            double (*av)[kSkNativeRows], int lane) {
  const int64_t chunks = (a.n + 31) / 32, total = (nr + kSkNativeRows - 1) / kSkNativeRows * chunks;
  const int64_t i1 = total * (worker + 1) / workers;
  int64_t i = total * worker / workers;
  int64_t g = i / chunks, c = i - g * chunks, prev = -1;
  const int k = static_cast<int>(a.k);
  for (; i < i1; ++i) {
    if (g != prev) {
      prev = g;
      __syncwarp();
      for (int x = lane; x < k * kSkNativeRows; x += 32) {
        const int64_t at = g * kSkNativeRows + x % kSkNativeRows;
        av[x / kSkNativeRows][x % kSkNativeRows] = at < nr ? a.fb.A[a.fb.rows[at] + x / kSkNativeRows * a.fb.lda] : 0.0;
      }
      __syncwarp();
    }
    const int64_t col = 32 * c + lane;
    const double* bp = a.fb.B + (col < a.n ? col : a.n - 1) * a.fb.ldb;
    double acc[kSkNativeRows], b[8];
#pragma unroll
    for (int r = 0; r < kSkNativeRows; ++r) acc[r] = 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) b[j] = j < k ? __ldg(bp + j) : 0.0;
    for (int l0 = 0; l0 < k; l0 += 8) {
      double next[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) next[j] = l0 + 8 + j < k ? __ldg(bp + l0 + 8 + j) : 0.0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (l0 + j < k) {
#pragma unroll
          for (int r = 0; r < kSkNativeRows; ++r) acc[r] = fma(av[l0 + j][r], b[j], acc[r]);
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) b[j] = next[j];
    }
#pragma unroll
    for (int r = 0; r < kSkNativeRows; ++r) {
      const int64_t at = g * kSkNativeRows + r;
      if (at < nr && col < a.n) a.C[a.fb.rows[at] + col * a.ldc] = acc[r];
    }
    if (++c == chunks) {
      c = 0;
      ++g;
    }
  }
}

// WIDE: |X| may reach 2^127 (r ≥ 14).
template <bool WIDE>
__global__ void __launch_bounds__(kSkThreads, 1)
    short_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, ShortArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sm_a = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sm_b = sm_a + kSkDigits * kTileBytes + kSkPad;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm_b + kSkStages * kSkStageStep);
  // bars: b_full[kSkStages], b_empty[kSkStages], acc_full[2], acc_empty[2], a_full, a_empty, drain
  __shared__ uint32_t tmem_base_s;
  __shared__ int na_s, nb_s;
  __shared__ __align__(16) double native_s[kSkNativeWarps][kSkK][kSkNativeRows];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bfull = smem_u32(bars), bempty = smem_u32(bars + kSkStages);
  const uint32_t accf = smem_u32(bars + 2 * kSkStages), acce = accf + 16, afull = accf + 32, aempty = accf + 40,
                 drain_bar = accf + 48;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSkStages; ++s) {
      mbar_init(bfull + 8 * s, 1);
      mbar_init(bempty + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf + 8 * b, 1);
      mbar_init(acce + 8 * b, kSkEpiWarps / 2);
    }
    mbar_init(afull, 1);
    mbar_init(aempty, 1);
    mbar_init(drain_bar, 1);
    fence_barrier_init();
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmB);
    na_s = nb_s = 1;
  }
  for (int i = threadIdx.x; i < (kSkStages + 1) * kSkPad / 16; i += kSkThreads) {
    const int stage = i / (kSkPad / 16), at = i % (kSkPad / 16);
    *reinterpret_cast<uint4*>(sm_b - kSkPad + stage * kSkStageStep + 16 * at) = make_uint4(0u, 0u, 0u, 0u);
  }
  fence_proxy_async_smem();  // the tensor core reads the pads
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_s), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  pdl_wait();  // the digits are written
  int na = 1, nb = 1;  // digits of A and B: the most any of their blocks needs
  for (int64_t i = threadIdx.x; i < a.nrb; i += kSkThreads) na = max(na, a.na[i]);
  for (int64_t i = threadIdx.x; i < a.nbb; i += kSkThreads) nb = max(nb, a.nb[i]);
  na = __reduce_max_sync(0xffffffffu, na);
  nb = __reduce_max_sync(0xffffffffu, nb);
  if (lane == 0) {
    atomicMax(&na_s, na);
    atomicMax(&nb_s, nb);
  }
  __syncthreads();
  {
    const DigitCounts dc = digit_counts(na_s, nb_s);
    na = __reduce_max_sync(0xffffffffu, dc.a);  // the same in every lane, and known to be
    nb = __reduce_max_sync(0xffffffffu, dc.b);
  }
  // This CTA's tiles: a contiguous range, row block by row block.
  const int64_t total = a.nrb * a.nct;
  const int64_t t0 = total * blockIdx.x / gridDim.x, t1 = total * (blockIdx.x + 1) / gridDim.x;
  // Row block and column tile of t0; the roles count on from there (a 64-bit
  // division per tile was most of a tile's time).
  const int nct = static_cast<int>(a.nct);
  const int first_rb = static_cast<int>(t0 / nct), first_ct = static_cast<int>(t0 - static_cast<int64_t>(first_rb) * nct);
  bool ok = true;
  // Flagged rows that this kernel's FP64 warps take: all of them or none.
  const int native = a.fb.count && *a.fb.count <= a.fb.most ? *a.fb.count : 0;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      int rb = first_rb, ct = first_ct, prev = -1;
      uint32_t it = 0, aph = 1, nblk = 0;
      for (int64_t t = t0; t < t1 && ok; ++t, ++it) {
        if (rb != prev) {
          if (!mbar_wait_bounded(aempty, aph, kWaitLimit)) {
            ok = false;
            break;
          }
          aph ^= 1;
          prev = rb;
          ++nblk;
          mbar_arrive_expect_tx(afull, static_cast<uint32_t>(na) * kTileBytes);
          for (int i = 0; i < na; ++i)
            tma_load_2d(smem_u32(sm_a + i * kTileBytes), &tmA, afull, 0, (rb * kSkDigits + i) * kRows);
        }
        const uint32_t s = it % kSkStages;
        if (!mbar_wait_bounded(bempty + 8 * s, ((it / kSkStages) & 1) ^ 1, kWaitLimit)) {
          ok = false;
          break;
        }
        mbar_arrive_expect_tx(bfull + 8 * s, kTileBytes);
        tma_load_2d(smem_u32(sm_b + s * kSkStageStep), &tmB, bfull + 8 * s, 0, ct * kRows);
        if (++ct == nct) {
          ct = 0;
          ++rb;
        }
      }
      if (!ok) {
        a.dev->status = kStatusTimeout;
        a.dev->timeout_site = 11;
      }
      // Every load has landed before the block leaves.
      for (uint32_t j = (it > kSkStages ? it - kSkStages : 0); j < it; ++j)
        mbar_wait_bounded(bfull + 8 * (j % kSkStages), (j / kSkStages) & 1, kWaitLimit);
      if (nblk) mbar_wait_bounded(afull, (nblk - 1) & 1, kWaitLimit);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    // One warp for both buffers: two, each with its own buffer, made the
    // tensor core alternate between them (2.41 against 2.31 ms, k = 64).
    const uint32_t me = lane == 0;
    // The f16 formats have the f8 descriptor's codes.
    auto idesc = [](int digits) { return idesc_f8_f32(kRows, kSkCols * digits); };
    constexpr uint64_t kDigitStep = kSkCols * kPlaneLine >> 4;  // one digit's lines of a B tile
    const uint64_t da = smem_desc_sw128(smem_u32(sm_a)), db = smem_desc_sw128(smem_u32(sm_b));
    auto run = [&](auto ksteps_c) {
      constexpr int KS = decltype(ksteps_c)::value;
      int ct = first_ct;
      uint32_t it = 0, aph = 0;
      bool fresh = true;  // a new row block: its digits have to land first
      for (int64_t t = t0; t < t1; ++t, ++it) {
        const uint32_t s = it % kSkStages, buf = it & 1;
        if ((fresh && !mbar_wait_bounded(afull, aph, kWaitLimit)) ||
            !mbar_wait_bounded(bfull + 8 * s, (it / kSkStages) & 1, kWaitLimit) ||
            !mbar_wait_bounded(acce + 8 * buf, ((it >> 1) & 1) ^ 1, kWaitLimit))
          ok = false;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (fresh) aph ^= 1;
        fresh = false;
        tc_fence_after();
        const uint64_t b = db + s * (kSkStageStep >> 4);
        const uint32_t acc0 = tmem + buf * kSkBufCols;
        // Digits i0 .. i0 + gd - 1 of A add to the weights i0 .. i0 + gd + nb
        // - 2, each with B's tile shifted by its place in the group (zero
        // lines come in at the ends).  The first product overwrites the
        // weights no earlier group has met and adds to the others.
        for (int i0 = 0; i0 < na; i0 += kSkGroup) {
          const int gd = min(kSkGroup, na - i0);
          const uint32_t acc = acc0 + i0 * kSkCols, all = idesc(nb + gd - 1);
          const uint64_t ag = da + i0 * (kTileBytes >> 4);
          if (i0 == 0) {
            mma_f16_by(me, acc, ag, b, all, 0u);
          } else {
            mma_f16_by(me, acc + (nb - 1) * kSkCols, ag, b + (nb - 1) * kDigitStep, idesc(gd), 0u);
            if (nb > 1) mma_f16_by(me, acc, ag, b, idesc(nb - 1), 1u);
          }
#pragma unroll
          for (int i = 0; i < kSkGroup; ++i) {
            if (i < gd) {
#pragma unroll
              for (int kk = i == 0 ? 1 : 0; kk < KS; ++kk)
                mma_f16_by(me, acc, ag + i * (kTileBytes >> 4) + 2 * kk, b - i * kDigitStep + 2 * kk, all, 1u);
            }
          }
        }
        mma_commit_by(me, bempty + 8 * s);
        mma_commit_by(me, accf + 8 * buf);
        if (++ct == nct) {
          ct = 0;
          fresh = true;
          mma_commit_by(me, aempty);  // the row block's digits are free
        }
      }
    };
    if (a.ksteps == 4) run(std::integral_constant<int, 4>());
    else if (a.ksteps == 3) run(std::integral_constant<int, 3>());
    else if (a.ksteps == 2) run(std::integral_constant<int, 2>());
    else run(std::integral_constant<int, 1>());
    if (!ok && lane == 0) {
      a.dev->status = kStatusTimeout;
      a.dev->timeout_site = 12;
    }
    mma_commit_by(me, drain_bar);  // every MMA retired before the tensor memory goes away
    mbar_wait_bounded(drain_bar, 0, kWaitLimit);
    __syncwarp();
  } else if (warp >= 2 + kSkEpiWarps) {
    // ---------------- native FP64 rows ----------------
    const int w = warp - 2 - kSkEpiWarps;
    if (native > 0)
      native_rows(a, native, static_cast<int>(blockIdx.x) * kSkNativeWarps + w, static_cast<int>(gridDim.x) * kSkNativeWarps,
                  native_s[w], lane);
  } else {
    // ---------------- epilogue ----------------
    // Warps 2..9 take the even tiles (buffer 0), 10..17 the odd ones, so that
    // one group's tensor-memory loads overlap the other's arithmetic; a warp
    // has 32 rows × 8 columns, four at a time.
    const uint32_t buf = (warp - 2) >> 3;
    const int q = warp & 3, h = ((warp - 2) & 7) >> 2;
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(32 * q) << 16) + buf * kSkBufCols + static_cast<uint32_t>(8 * h);
    auto run = [&](auto weights_c) {
      constexpr int W = decltype(weights_c)::value;  // weights in use
      int rb = first_rb, ct = first_ct + static_cast<int>(buf), prev = -1;
      uint32_t ph = 0;
      int dr = 0;
      bool live = false;  // the row exists, and no FP64 warp has it
      for (int64_t t = t0 + buf; t < t1; t += 2, ct += 2, ph ^= 1) {
        for (; ct >= nct; ct -= nct) ++rb;
        const int64_t row = static_cast<int64_t>(rb) * kRows + 32 * q + lane;
        if (rb != prev) {
          prev = rb;
          dr = row < a.m ? __ldg(a.d + row) : 0;
          live = row < a.m && !(native > 0 && (__ldg(a.fb.flag + row) & 1));
        }
        // The columns' exponents, four ahead of their use (past n: within the
        // array's 256-byte slot).
        const int4* ep = reinterpret_cast<const int4*>(a.e + static_cast<int64_t>(ct) * kSkCols + 8 * h);
        int4 next_e = __ldg(ep);
        if (!mbar_wait_bounded(accf + 8 * buf, ph, kWaitLimit)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const bool whole = live && (ct + 1) * static_cast<int64_t>(kSkCols) <= a.n;
        double* cp = a.C + row + (static_cast<int64_t>(ct) * kSkCols + 8 * h) * a.ldc;
#pragma unroll 1
        for (int c = 0; c < 8; c += 4) {
          const int64_t col = static_cast<int64_t>(ct) * kSkCols + 8 * h + c;
          const int ec[4] = {next_e.x, next_e.y, next_e.z, next_e.w};
          if (c == 0) next_e = __ldg(ep + 1);
          uint32_t v[W][4];
#pragma unroll
          for (int w = 0; w < W; ++w) tmem_ld4(lane_addr + c + w * kSkCols, v[w]);
          tmem_ld_wait();
          if (c == 4) {  // the buffer is free (relaxed: the stores of C need no ordering against the MMAs)
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_relaxed(acce + 8 * buf);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // Four weights to a 64-bit sum (below 2^48) on top of the carry of
            // the four before: a 32-bit word of X each.
            uint32_t x[4];
            int carry = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              long long s = carry;
#pragma unroll
              for (int i = 0; i < 4; ++i)
                if (4 * g + i < W) s = mad_wide(__float2int_rn(__uint_as_float(v[4 * g + i][j])), a.pow256[i], s);
              x[g] = static_cast<uint32_t>(s);
              carry = static_cast<int>(s >> 32);
            }
            const int E = -(dr + ec[j]);
            double val;
            if (WIDE && carry != static_cast<int>(x[3]) >> 31)
              val = finish_signed_slow(static_cast<uint32_t>(carry), x[3], x[2], x[1], x[0], E);
            else
              val = finish_signed(x[3], x[2], x[1], x[0], E);
            if (whole || (live && col + j < a.n)) *cp = val;
            cp += a.ldc;
          }
        }
      }
    };
    const int weights = na + nb - 1;
    if (weights > 12) run(std::integral_constant<int, kSkClasses>());
    else if (weights > 8) run(std::integral_constant<int, 12>());
    else if (weights > 4) run(std::integral_constant<int, 8>());
    else run(std::integral_constant<int, 4>());
    if (!ok) {
      a.dev->status = kStatusTimeout;
      a.dev->timeout_site = 13;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

static size_t short_smem() {
  return 1024 + kSkDigits * static_cast<size_t>(kTileBytes) + kSkPad + kSkStages * static_cast<size_t>(kSkStageStep) + 8 * (2 * kSkStages + 7);
}

// Scratch: A's digit lines, B's, then the digit counts.
struct ShortScratch {
  size_t b_off, na_off, nb_off, total;
};
static ShortScratch short_scratch(int64_t m, int64_t n) {
  const int64_t mb = (m + kRows - 1) / kRows, ct = (n + kSkCols - 1) / kSkCols, nb = (n + kRows - 1) / kRows;
  ShortScratch s;
  s.b_off = static_cast<size_t>(mb) * kSkDigits * kTileBytes;
  s.na_off = s.b_off + static_cast<size_t>(ct) * kTileBytes;
  s.nb_off = s.na_off + sizeof(int) * static_cast<size_t>(mb);
  s.total = s.nb_off + sizeof(int) * static_cast<size_t>(nb);
  return s;
}

// The digits of both operands, 1 KiB a row or column, fit where the digit
// planes would go from r = 4 on (8 planes of 128 bytes); the line coordinates
// of the tensor maps are 32-bit.
bool short_k_applies(int64_t m, int64_t n, int64_t k, size_t scratch_bytes) {
  return k <= kSkK && m <= (int64_t{1} << 26) && n <= (int64_t{1} << 26) && short_scratch(m, n).total <= scratch_bytes;
}

cudaError_t launch_short_digits(int64_t m, int64_t n, int64_t k, const double* A, int64_t lda, const double* B,
                                int64_t ldb, const int32_t* ra, const int32_t* cb, const int32_t* d, const int32_t* e,
                                const uint8_t* row_flag, const uint8_t* col_flag, uint8_t* scratch, cudaStream_t st) {
  const ShortScratch sc = short_scratch(m, n);
  const int64_t mb = (m + kRows - 1) / kRows, nb = (n + kRows - 1) / kRows;
  const DigitOperand xa{A, 1, lda, m, mb * kRows, d, ra, row_flag, scratch, reinterpret_cast<int*>(scratch + sc.na_off)};
  const DigitOperand xb{B,        ldb,           1, n, (n + kSkCols - 1) / kSkCols * kSkCols, e, cb, col_flag,
                        scratch + sc.b_off, reinterpret_cast<int*>(scratch + sc.nb_off)};
  count_launch();
  return launch_dependent(short_digits_kernel, dim3(static_cast<unsigned>(mb + nb)), dim3(kSkDigitThreads), 0, st, xa,
                          xb, mb, k);
}

static int64_t short_grid(int64_t m, int64_t cols) {
  return std::min<int64_t>(num_sms(), (m + kRows - 1) / kRows * ((cols + kSkCols - 1) / kSkCols));
}

// The flagged rows that the FP64 warps take: as many as they finish before the
// products and the fallback kernel after them would.  Two warps of a CTA run 1 G
// FMAs a second, the fallback kernel, on all of the FP64 pipe, 0.55 T after 30 µs
// of its own, and the products 140 G outputs.  16384²×64, a call with 16, 164,
// 400, 512 flagged rows: 2377, 2707, 3136, 3288 µs with the fallback kernel,
// 2182, 2198, 2791, 3378 with these warps; 2048²×64 with 64: 140 and 89;
// 20000×100×64 with 600: 139 and 76; 128²×64 with 1: 69 and 40.
int short_native_rows(int64_t m, int64_t n, int64_t k) {
  const double fmas = static_cast<double>((n + 31) / 32 * 32) * static_cast<double>(k);  // a row's, in whole warps
  const double extra = 1e-9 / static_cast<double>(short_grid(m, n)) - 1 / 0.55e12;
  const double rows = (static_cast<double>(m) * static_cast<double>(n) / 140e9 + 30e-6) / (fmas * extra);
  return static_cast<int>(std::min(rows, 1e6));
}

// Columns [c0, c0 + cols) of C (c0 a multiple of 128; C, e at column c0).
cudaError_t launch_short_gemm(int64_t m, int64_t n, int64_t k, int64_t c0, int64_t cols, int T, const uint8_t* scratch,
                              const int32_t* d, const int32_t* e, double* C, int64_t ldc, const NativeRows& fb,
                              Oz2Device* dev, cudaStream_t st) {
  const ShortScratch sc = short_scratch(m, n);
  ShortArgs a{};
  a.m = m;
  a.n = cols;
  a.nrb = (m + kRows - 1) / kRows;
  a.nct = (cols + kSkCols - 1) / kSkCols;
  a.nbb = (n + kRows - 1) / kRows;
  a.ldc = ldc;
  a.ksteps = static_cast<int>((k + 15) / 16);
  a.na = reinterpret_cast<const int*>(scratch + sc.na_off);
  a.nb = reinterpret_cast<const int*>(scratch + sc.nb_off);
  a.d = d;
  a.e = e;
  a.C = C;
  a.dev = dev;
  a.fb = fb;
  a.k = k;
  for (int i = 0; i < 4; ++i) a.pow256[i] = 1 << (8 * i);
  CUtensorMap ta, tb;
  if (!make_block_map(&ta, scratch, m, kPlaneLine, kSkDigits) ||
      !make_block_map(&tb, scratch + sc.b_off + static_cast<size_t>(c0 / kSkCols) * kTileBytes, a.nct * kRows, kPlaneLine, 1))
    return cudaErrorInvalidValue;
  auto kern = T > 125 ? short_gemm_kernel<true> : short_gemm_kernel<false>;
  const size_t smem = short_smem();
  const cudaError_t err = allow_smem(reinterpret_cast<const void*>(kern), smem);
  if (err != cudaSuccess) return err;
  count_launch();
  const int64_t grid = short_grid(m, cols);
  return launch_dependent(kern, dim3(static_cast<unsigned>(grid)), dim3(kSkThreads), smem, st, ta, tb, a);
}

}  // namespace oz2
