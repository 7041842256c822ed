// C for a skinny product (few columns or few rows of C, a long k) without
// digit planes and residues: the products of the scaled integers' base-256
// digits, as for a short k (k_short.cu), with the tall operand's digits formed
// on chip.
//
// For a C of a few columns every element of A feeds one tile column, so the
// residue path's time is storing and reading back A's digit planes
// (16384×16×16384, r = 12: 2.03 ms to write 8 GB, 1.36 ms to read them).  Here
// A is read once per 16 columns and nothing of it is written: a thread
// quantises 8 entries of a row (Eq. scale), writes their balanced base-256
// digits, up to 8, as f16 operand tiles to shared memory, and one MMA per digit
// adds its products with every digit of the skinny operand to the accumulators
// of their weights.  The sums of 128 k-entries stay exact in FP32 (8 digit pairs
// · 128 · 2^14 = 2^24); the accumulators are then added to the integer X_ij that
// a thread keeps in registers, 160 bits wide, while the tensor core goes on in
// the other buffer.  X is the integer the CRT would return, rounded alike: the
// same bits of C.
//
// The work, (16 columns, 128 rows, 128 k-entries) slabs, is dealt to the CTAs
// in equal contiguous runs, whatever the shape; the parts of an output's sum
// that different CTAs form meet in scratch, where skinny_finish_kernel adds and
// rounds them.
//
// With few rows of C instead, B takes A's place (its columns are the rows).
//
// Measured on one GB300, 16384×16×16384, r = 12 (seven digits of A): 0.72 ms
// for this kernel (2.15 GB read once, 0.32 ms at the copy rate) against 2.03 +
// 1.36 for the planes; the call 4.32 → 1.39 ms, the "+1" pass below included.
// The converting warps' integer pipe bounds it (62 instructions per entry, 60%
// busy, the loads' latency next: a second chunk in flight spills at the 96
// registers 18 warps allow and is slower).
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "oz2_crt.cuh"
#include "oz2_gemm.cuh"
#include "oz2_quant.cuh"

namespace oz2 {

constexpr int kSnDigits = 8;                          // base-256 digits of an integer below 2^62
constexpr int kSnCols = 16;                           // columns of the skinny operand per pass
constexpr int kSnK = 32;                              // k-entries of a chunk (two MMA K-steps)
constexpr int kSnSlabChunks = 4;                      // chunks summed in FP32: 128 k-entries
constexpr int kSnGroup = 4;                           // digits that share an accumulator window (k_short.cu)
constexpr int kSnClasses = 2 * kSnDigits - 1;
constexpr int kSnATile = kRows * 16 + 32;             // 128 rows × 8 entries: a K column of core matrices (and a
                                                      // bank offset: lanes that hold four K columns of a row)
constexpr int kSnADigit = kSnATile * (kSnK / 8);      // 8 KiB: a digit of a chunk
constexpr int kSnABuf = kSnDigits * kSnADigit;        // 64 KiB
constexpr int kSnPad = (kSnGroup - 1) * kSnCols;      // zero rows on both sides of the skinny operand's digits
constexpr int kSnBRows = kSnDigits * kSnCols + 2 * kSnPad;  // 224
constexpr int kSnBTile = kSnBRows * 16;
constexpr int kSnBChunk = kSnBTile * (kSnK / 8);      // 14 KiB
constexpr int kSnBStages = 4;
constexpr int kSnBufCols = 256;
constexpr int kSnWarps = 16;                          // conversion and sums
constexpr int kSnThreads = 32 * (kSnWarps + 2);       // MMA issuer, loads of the skinny operand
constexpr int kSnOutputs = kRows * kSnCols;           // outputs of a (row block, column group)
constexpr int kSnWords = 5;                           // 160-bit sums

struct SkinnyArgs {
  const double* T;                  // the tall operand: entry (row, l) at row·row_stride + l·k_stride
  int64_t row_stride, k_stride, rows, k;
  int64_t nrb, slabs, total;        // row blocks, slabs of k, (column group, row block, slab) units
  const int32_t *exps, *scan;       // d and ra (e and cb when B is tall)
  const uint8_t* flag;
  const int32_t *s_exps, *s_scan;   // of the skinny operand
  const uint8_t* s_flag;
  int64_t cols;                     // its columns
  const uint8_t* digits;            // its digit chunks: [group][chunk][kSnBChunk]
  int vec;                          // rows contiguous in k and 16-byte aligned
  uint32_t* parts;                  // [group·row block][slot][word][column][row]
  int slots;
  Oz2Device* dev;
  int pow256[4];                    // as data: see short_gemm_kernel
};

// CTA that takes unit u of `total` dealt to `grid` CTAs in runs [total·c/grid, total·(c+1)/grid).
__host__ __device__ __forceinline__ int64_t cta_of(int64_t u, int64_t total, int64_t grid) {
  return ((u + 1) * grid - 1) / total;
}

// ---------------------------------------------------------------------------
// Digits of the skinny operand: f16 operand tiles of 8-row × 16-byte core
// matrices, chunk by chunk, 48 zero rows before and after the 16 columns of
// digit 0, of digit 1, and so on.  A thread takes 8 entries of a column.
// ---------------------------------------------------------------------------
// Digits 4·half .. 4·half + 3 of 8 entries as halves (lo[e] holds those digits
// plus 128 as bytes): byte pairs of neighbouring entries, made 1024 + byte by a
// byte permute, less 1152.
template <class Store>
__device__ __forceinline__ void digit_halves(const uint32_t (&word)[8], Store store) {
  uint32_t h[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t p01 = __byte_perm(word[2 * j], word[2 * j + 1], 0x5140), p23 = __byte_perm(word[2 * j], word[2 * j + 1], 0x7362);
    h[0][j] = __byte_perm(p01, 0x64646464u, 0x4140);
    h[1][j] = __byte_perm(p01, 0x64646464u, 0x4342);
    h[2][j] = __byte_perm(p23, 0x64646464u, 0x4140);
    h[3][j] = __byte_perm(p23, 0x64646464u, 0x4342);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&h[i][j]), __half2half2(__ushort_as_half(0x6480)));
      w[j] = *reinterpret_cast<const uint32_t*>(&v);
    }
    store(i, make_uint4(w[0], w[1], w[2], w[3]));
  }
}
constexpr unsigned long long kDigitBias = 0x8080808080808080ull;  // digits -128..127 as bytes 0..255

// Ã + kDigitBias for a truncated entry of a row with d ≤ kTzFastMaxD, as
// quantise_tz forms Ã (rb = 1085 - d): one 64-bit shift, which clamps, and the
// sign's last bit taken in with the bias.
__device__ __forceinline__ void quantise_tz_biased(double x, int rb, uint32_t& lo_out, uint32_t& hi_out) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const uint32_t E = (hi >> 20) & 0x7FFu;
  const uint32_t mh = (min(E, 1u) << 20) + (hi & 0xFFFFFu);
  const uint32_t r = static_cast<uint32_t>(rb) - max(E, 1u);
  const unsigned long long m = (static_cast<unsigned long long>(__funnelshift_l(lo, mh, 10)) << 32) | (lo << 10);
  unsigned long long q;
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(m), "r"(r));
  const uint32_t sgn = static_cast<uint32_t>(static_cast<int>(hi) >> 31);  // 0 or all ones
  const unsigned long long t = ((static_cast<unsigned long long>(static_cast<uint32_t>(q >> 32) ^ sgn) << 32) |
                                (static_cast<uint32_t>(q) ^ sgn)) +
                               ((0x80808080ull << 32) | (0x80808080u - sgn));
  lo_out = static_cast<uint32_t>(t);
  hi_out = static_cast<uint32_t>(t >> 32);
}

__global__ void __launch_bounds__(256) skinny_digits_kernel(const double* __restrict__ S, int64_t col_stride,
                                                            int64_t k_stride, int64_t cols, int64_t k,
                                                            const int32_t* __restrict__ exps,
                                                            const uint8_t* __restrict__ flag, int64_t chunks,
                                                            int64_t groups, uint8_t* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int c = static_cast<int>(idx % kSnCols);
  const int64_t oct = idx / kSnCols, per_group = chunks * (kSnK / 8);
  if (oct >= per_group * groups) return;
  const int64_t g = oct / per_group, l0 = (oct - g * per_group) * 8;
  const int64_t col = g * kSnCols + c;
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) lo[j] = hi[j] = 0x80808080u;
  if (col < cols && !(flag[col] & 2)) {
    const int e = exps[col];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (l0 + j < k) {
        const unsigned long long u = quantise_entry(__ldg(S + col * col_stride + (l0 + j) * k_stride), e, false) + kDigitBias;
        lo[j] = static_cast<uint32_t>(u);
        hi[j] = static_cast<uint32_t>(u >> 32);
      }
  }
  uint8_t* dst = out + oct * kSnBTile;  // 8 entries: one K column of core matrices
  auto put = [&](int i, uint4 v) { *reinterpret_cast<uint4*>(dst + (kSnPad + i * kSnCols + c) * 16) = v; };
  digit_halves(lo, [&](int i, uint4 v) { put(i, v); });
  digit_halves(hi, [&](int i, uint4 v) { put(4 + i, v); });
#pragma unroll
  for (int p = c; p < kSnPad; p += kSnCols) {
    *reinterpret_cast<uint4*>(dst + p * 16) = make_uint4(0u, 0u, 0u, 0u);
    *reinterpret_cast<uint4*>(dst + (kSnBRows - 1 - p) * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// ---------------------------------------------------------------------------
// The products.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mma_f8_by(uint32_t me, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(me)
      : "memory");
}
// Linear copy of global memory into shared memory, completing on an mbarrier
// (16-byte aligned, a multiple of 16 bytes).
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t (&v)[2]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(taddr));
}

// KMAJOR: the tall operand's rows are contiguous in k (columns of B); its
// entries are then loaded by four lanes a row, otherwise (A) by a lane a row.
template <bool KMAJOR>
__global__ void __launch_bounds__(kSnThreads, 1) skinny_kernel(const __grid_constant__ SkinnyArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sm_a = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sm_b = sm_a + 2 * kSnABuf;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm_b + kSnBStages * kSnBChunk);
  __shared__ uint32_t tmem_base_s;
  __shared__ int na_s, nb_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t afull = smem_u32(bars), aempty = afull + 16, accf = afull + 32, acce = afull + 48,
                 bfull = afull + 64, bempty = bfull + 8 * kSnBStages, drain_bar = bempty + 8 * kSnBStages;
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(afull + 8 * b, kSnWarps);
      mbar_init(aempty + 8 * b, 1);
      mbar_init(accf + 8 * b, 1);
      mbar_init(acce + 8 * b, kSnWarps);
    }
    for (int s = 0; s < kSnBStages; ++s) {
      mbar_init(bfull + 8 * s, 1);
      mbar_init(bempty + 8 * s, 1);
    }
    mbar_init(drain_bar, 1);
    fence_barrier_init();
    na_s = nb_s = 1;
  }
  if (warp == kSnWarps) {
    tmem_alloc(smem_u32(&tmem_base_s), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  pdl_wait();  // exponents, flags and the skinny operand's digits
  const int64_t u0 = a.total * blockIdx.x / gridDim.x, u1 = a.total * (blockIdx.x + 1) / gridDim.x;
  const int64_t first_q = u0 / a.slabs, last_q = (u1 - 1) / a.slabs;  // column group · row blocks + row block
  // Digits this CTA needs: |Ã| ≤ 2^t for t = scale + max-exponent, and n digits
  // hold ±2^(8n - 2).
  {
    int need = 1;
    for (int64_t q = first_q; q <= last_q; ++q) {
      const int64_t row = (q % a.nrb) * kRows + threadIdx.x;
      if (threadIdx.x < kRows && row < a.rows && !(a.flag[row] & 2))
        need = max(need, min(kSnDigits, (a.exps[row] + a.scan[row] + 9) >> 3));
    }
    atomicMax(&na_s, need);
    need = 1;
    for (int64_t c = threadIdx.x; c < a.cols; c += kSnThreads)
      if (!(a.s_flag[c] & 2)) need = max(need, min(kSnDigits, (a.s_exps[c] + a.s_scan[c] + 9) >> 3));
    atomicMax(&nb_s, need);
  }
  __syncthreads();
  // Thirteen weights, which r = 12 needs, or all fifteen.  The digits added are
  // zero: the skinny operand's first, since the tall one's are formed here.
  // (With twelve or fifteen, the tall operand's first, 16384×16×16384 r = 12
  // 1.433 ms a call against 1.387, 9000×16×9000 r = 6 0.485 against 0.463.)
  int na = na_s, nb = nb_s;
  if (na + nb - 1 <= 13) {
    const int more = 14 - na - nb;
    const int x = min(kSnDigits, nb + more);  // the skinny operand's: its tiles hold all eight
    na += nb + more - x;
    nb = x;
  } else {
    na = nb = kSnDigits;
  }
  na = __reduce_max_sync(0xffffffffu, na);  // the same in every lane, and known to be
  nb = __reduce_max_sync(0xffffffffu, nb);
  const int units = static_cast<int>(u1 - u0);
  bool ok = true;

  if (warp == kSnWarps + 1) {
    // ---------------- the skinny operand's chunks ----------------
    if (lane == 0) {
      int64_t slab = u0 - first_q * a.slabs, q = first_q;
      const int64_t group_bytes = a.slabs * kSnSlabChunks * kSnBChunk;
      uint32_t it = 0;
      for (int t = 0; t < units && ok; ++t) {
        const uint8_t* src = a.digits + (q / a.nrb) * group_bytes + slab * kSnSlabChunks * kSnBChunk;
        for (int c = 0; c < kSnSlabChunks; ++c, ++it) {
          const uint32_t s = it % kSnBStages;
          if (!mbar_wait_bounded(bempty + 8 * s, ((it / kSnBStages) & 1) ^ 1, kWaitLimit)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(bfull + 8 * s, kSnBChunk);
          bulk_load(smem_u32(sm_b + s * kSnBChunk), src + c * kSnBChunk, kSnBChunk, bfull + 8 * s);
        }
        if (++slab == a.slabs) {
          slab = 0;
          ++q;
        }
      }
      if (!ok) {
        a.dev->status = kStatusTimeout;
        a.dev->timeout_site = 14;
      }
      // Every load has landed before the block leaves.
      for (uint32_t j = (it > kSnBStages ? it - kSnBStages : 0); j < it; ++j)
        mbar_wait_bounded(bfull + 8 * (j % kSnBStages), (j / kSnBStages) & 1, kWaitLimit);
    }
    __syncwarp();
  } else if (warp == kSnWarps) {
    // ---------------- MMA issuer (the warp runs, lane 0 issues) ----------------
    const uint32_t me = lane == 0;
    auto idesc = [](int digits) { return idesc_f8_f32(kRows, kSnCols * digits); };  // the f16 formats have the f8 codes
    constexpr uint64_t kDigitStep = kSnCols * 16 >> 4;
    const uint64_t da = smem_desc_plain(smem_u32(sm_a), kSnATile, 128);
    const uint64_t db = smem_desc_plain(smem_u32(sm_b) + kSnPad * 16, kSnBTile, 128);
    uint32_t it = 0;
    for (int t = 0; t < units && ok; ++t) {
      const uint32_t buf = t & 1, acc0 = tmem + buf * kSnBufCols;
      ok = mbar_wait_warp(acce + 8 * buf, ((t >> 1) & 1) ^ 1, kWaitLimit);
#pragma unroll 1
      for (int c = 0; c < kSnSlabChunks && ok; ++c, ++it) {
        const uint32_t b = it & 1, s = it % kSnBStages;
        ok = mbar_wait_warp(afull + 8 * b, (it >> 1) & 1, kWaitLimit) &&
             mbar_wait_warp(bfull + 8 * s, (it / kSnBStages) & 1, kWaitLimit);
        if (!ok) break;
        tc_fence_after();
        const uint64_t ab = da + b * (kSnABuf >> 4), bb = db + s * (kSnBChunk >> 4);
        // Two windows of four digits each (see k_short.cu), the second first
        // in odd chunks: the accumulator window moves once a chunk.
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int i0 = (half ^ (c & 1)) * kSnGroup;
          const int gd = min(kSnGroup, na - i0);
          if (gd <= 0) continue;
          const uint32_t acc = acc0 + i0 * kSnCols, all = idesc(nb + gd - 1);
          const uint64_t ag = ab + i0 * (kSnADigit >> 4);
          if (c == 0) {  // the slab's first products: overwrite the weights met for the first time
            if (i0 == 0) {
              mma_f16_by(me, acc, ag, bb, all, 0u);
            } else {
              mma_f16_by(me, acc + (nb - 1) * kSnCols, ag, bb + (nb - 1) * kDigitStep, idesc(gd), 0u);
              if (nb > 1) mma_f16_by(me, acc, ag, bb, idesc(nb - 1), 1u);
            }
          } else {
            mma_f16_by(me, acc, ag, bb, all, 1u);
          }
#pragma unroll
          for (int i = 0; i < kSnGroup; ++i) {
            if (i < gd) {
#pragma unroll
              for (int kk = i == 0 ? 1 : 0; kk < kSnK / 16; ++kk)
                mma_f16_by(me, acc, ag + i * (kSnADigit >> 4) + kk * (2 * kSnATile >> 4),
                       bb - i * kDigitStep + kk * (2 * kSnBTile >> 4), all, 1u);
            }
          }
        }
        mma_commit_by(me, aempty + 8 * b);
        mma_commit_by(me, bempty + 8 * s);
      }
      if (ok) mma_commit_by(me, accf + 8 * buf);
    }
    if (!ok && me) {
      a.dev->status = kStatusTimeout;
      a.dev->timeout_site = 15;
    }
    mma_commit_by(me, drain_bar);  // every MMA retired before the tensor memory goes away
    mbar_wait_bounded(drain_bar, 0, kWaitLimit);
    __syncwarp();
  } else {
    // ---------------- digits of the tall operand, and the sums ----------------
    const int rq = warp & 3, cq = warp >> 2;  // sums: rows 32·rq + lane, columns 4·cq .. 4·cq + 3
    // Digits: 8 entries (`part` of a chunk) of a row.
    const int rloc = KMAJOR ? 8 * warp + (lane >> 2) : 32 * rq + lane, part = KMAJOR ? lane & 3 : cq;
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(32 * rq) << 16) + static_cast<uint32_t>(4 * cq);
    auto run = [&](auto weights_c) {
      constexpr int W = decltype(weights_c)::value;
      uint32_t X[4][kSnWords];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int w = 0; w < kSnWords; ++w) X[j][w] = 0u;
      // Slab t of this CTA: its accumulators into X; after the last slab of a
      // row block (or of the CTA) X goes out.
      auto drain = [&](int t, bool out, int64_t q) {
        const uint32_t buf = t & 1;
        ok = mbar_wait_warp(accf + 8 * buf, (t >> 1) & 1, kWaitLimit);
        if (!ok) return;
        tc_fence_after();
#pragma unroll
        for (int j2 = 0; j2 < 4; j2 += 2) {
          uint32_t v[W][2];
#pragma unroll
          for (int w = 0; w < W; ++w) tmem_ld2(lane_addr + buf * kSnBufCols + w * kSnCols + j2, v[w]);
          tmem_ld_wait();
          if (j2 == 2) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_relaxed(acce + 8 * buf);
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            int carry = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              long long s = static_cast<long long>(carry) + static_cast<long long>(X[j2 + j][g]);
#pragma unroll
              for (int i = 0; i < 4; ++i)
                if (4 * g + i < W) s = mad_wide(__float2int_rn(__uint_as_float(v[4 * g + i][j])), a.pow256[i], s);
              X[j2 + j][g] = static_cast<uint32_t>(s);
              carry = static_cast<int>(s >> 32);
            }
            X[j2 + j][4] += static_cast<uint32_t>(carry);
          }
        }
        if (out) {
          const int64_t slot = blockIdx.x - cta_of(q * a.slabs, a.total, gridDim.x);
          uint32_t* dst = a.parts + (q * a.slots + slot) * (kSnWords * kSnOutputs) + 4 * cq * kRows + 32 * rq + lane;
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int w = 0; w < kSnWords; ++w) {
              dst[w * kSnOutputs + j * kRows] = X[j][w];
              X[j][w] = 0u;
            }
        }
      };
      int64_t q = first_q, slab = u0 - first_q * a.slabs;
      int d = 0;
      const double* p = nullptr;  // this thread's first entry of the slab
      auto enter = [&]() {        // a new row block
        const int64_t row = (q % a.nrb) * kRows + rloc;
        const bool live = row < a.rows && !(a.flag[row] & 2);
        d = live ? a.exps[row] : -4096;  // quantises any entry to zero
        p = a.T + (row < a.rows ? row : a.rows - 1) * a.row_stride;
      };
      // 8 entries of chunk c of slab `sl` (zero past k).
      auto fetch = [&](const double* base, int64_t sl, int c, double (&x)[8]) {
        const int64_t l = (sl * kSnSlabChunks + c) * kSnK + part * 8;
        const double* e = base + l * a.k_stride;
        if (KMAJOR && a.vec && l + 8 <= a.k) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const double2 v = __ldg(reinterpret_cast<const double2*>(e) + j);
            x[2 * j] = v.x;
            x[2 * j + 1] = v.y;
          }
        } else if (l + 8 <= a.k) {
#pragma unroll
          for (int j = 0; j < 8; ++j, e += a.k_stride) x[j] = __ldg(e);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j, e += a.k_stride) x[j] = l + j < a.k ? __ldg(e) : 0.0;
        }
      };
      enter();
      double x[8];
      fetch(p, slab, 0, x);
      uint32_t it = 0;
      bool out = false;     // slab t - 1 ended a row block, `out_q`
      int64_t out_q = 0;
      for (int t = 0; t < units && ok; ++t) {
        const int dt = d;
        const bool ends = slab + 1 == a.slabs;
        const int64_t qt = q;
#pragma unroll 1
        for (int c = 0; c < kSnSlabChunks; ++c, ++it) {
          uint32_t lo[8], hi[8];
          if (dt <= kTzFastMaxD) {
            const int rb = 1085 - dt;
#pragma unroll
            for (int j = 0; j < 8; ++j) quantise_tz_biased(x[j], rb, lo[j], hi[j]);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const unsigned long long u = quantise_entry(x[j], dt, false) + kDigitBias;
              lo[j] = static_cast<uint32_t>(u);
              hi[j] = static_cast<uint32_t>(u >> 32);
            }
          }
          // The next chunk's entries are in flight while this one is stored.
          if (c + 1 < kSnSlabChunks) {
            fetch(p, slab, c + 1, x);
          } else if (t + 1 < units) {
            if (ends) {
              slab = 0;
              ++q;
              enter();
            } else {
              ++slab;
            }
            fetch(p, slab, 0, x);
          }
          const uint32_t b = it & 1;
          ok = mbar_wait_warp(aempty + 8 * b, ((it >> 1) & 1) ^ 1, kWaitLimit);
          if (!ok) break;
          uint8_t* dst = sm_a + b * kSnABuf + part * kSnATile + rloc * 16;
          digit_halves(lo, [&](int i, uint4 v) {
            if (i < na) *reinterpret_cast<uint4*>(dst + i * kSnADigit) = v;
          });
          if (na > 4)
            digit_halves(hi, [&](int i, uint4 v) {
              if (4 + i < na) *reinterpret_cast<uint4*>(dst + (4 + i) * kSnADigit) = v;
            });
          fence_proxy_async_smem();  // the tensor core reads what the threads wrote
          __syncwarp();
          if (lane == 0) mbar_arrive(afull + 8 * b);
        }
        if (!ok) break;
        if (t > 0) drain(t - 1, out, out_q);
        out = ends || t + 1 == units;
        out_q = qt;
      }
      if (ok && units > 0) drain(units - 1, out, out_q);
    };
    if (na + nb - 1 <= 13) run(std::integral_constant<int, 13>());
    else run(std::integral_constant<int, kSnClasses>());
    if (!ok && lane == 0) {
      a.dev->status = kStatusTimeout;
      a.dev->timeout_site = 16;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kSnWarps) tmem_dealloc(tmem, 512);
}

// The parts of each output's sum, added and rounded into C.  Row r of the tall
// operand and column c of the skinny one: C at r·tall_stride + c·skinny_stride.
__global__ void __launch_bounds__(kRows) skinny_finish_kernel(const uint32_t* __restrict__ parts, int64_t slabs,
                                                              int64_t total, int64_t grid, int slots, int64_t nrb,
                                                              int64_t rows, int64_t cols,
                                                              const int32_t* __restrict__ exps,
                                                              const int32_t* __restrict__ s_exps, double* __restrict__ C,
                                                              int64_t tall_stride, int64_t skinny_stride) {
  pdl_trigger();
  pdl_wait();
  const int64_t q = blockIdx.x;
  const int64_t row = (q % nrb) * kRows + threadIdx.x, col = (q / nrb) * kSnCols + blockIdx.y;
  if (row >= rows || col >= cols) return;
  const int n = static_cast<int>(cta_of((q + 1) * slabs - 1, total, grid) - cta_of(q * slabs, total, grid)) + 1;
  const uint32_t* src = parts + q * slots * (kSnWords * kSnOutputs) + blockIdx.y * kRows + threadIdx.x;
  uint32_t x[kSnWords] = {};
  for (int s = 0; s < n; ++s, src += kSnWords * kSnOutputs) {
    unsigned long long t = 0;
#pragma unroll
    for (int w = 0; w < kSnWords; ++w) {
      t += static_cast<unsigned long long>(x[w]) + __ldg(src + w * kSnOutputs);
      x[w] = static_cast<uint32_t>(t);
      t >>= 32;
    }
  }
  const int E = -(exps[row] + s_exps[col]);
  double val;
  if (static_cast<int>(x[4]) != static_cast<int>(x[3]) >> 31)
    val = finish_signed_slow(x[4], x[3], x[2], x[1], x[0], E);
  else
    val = finish_signed(x[3], x[2], x[1], x[0], E);
  C[row * tall_stride + col * skinny_stride] = val;
}

// ---------------------------------------------------------------------------
// The "+1" pass (§2.4) of a product with few columns: U = ÂB̂ with A's magnitude
// codes formed on chip, instead of writing their plane and reading it back.  A
// thread makes the 16 codes of one core-matrix row; the tensor core sums all of
// a CTA's run of k in FP32 (every partial sum is an integer number of units
// below 2^24, so their order is free), and the runs add into U, whose row maxima
// plus_one_rowmax_kernel then takes.  The loads of A bound it: two CTAs an SM
// (one left a third of them unhidden).  Measured, 16384×16×16384: 0.35 ms for
// the plane and the GEMM's 0.47 + 0.05 (the call 1.59 → 1.44 ms).
// ---------------------------------------------------------------------------
constexpr int kSpK = 64;                               // k-entries of a chunk: two MMA K-steps
constexpr int kSpATile = kRows * 16;                   // 128 rows × 16 entries
constexpr int kSpABuf = kSpATile * (kSpK / 16);        // 8 KiB
constexpr int kSpABufs = 4;
constexpr int kSpColsMax = 80;                         // columns of the skinny operand, in sixteens
constexpr int kSpBBuf = kSpColsMax * kSpK;             // 5 KiB
constexpr int kSpCodeWarps = 16;
constexpr int kSpThreads = 32 * (kSpCodeWarps + 2);    // MMA issuer, copies of the skinny operand's codes

struct SkinnyPlusArgs {
  const double* A;
  int64_t lda, rows, k;
  int64_t nrb, chunks, total;     // row blocks, chunks of k, their product
  const int32_t* scan;
  const uint8_t* flag;
  int clamp;
  const uint8_t* codes;           // of B: cols × k_pad bytes
  int64_t cols, k_pad;
  int npad;                       // cols to a multiple of 16
  float* U;                       // row-major, ld = ldu
  int64_t ldu;
  Oz2Device* dev;
};

__global__ void __launch_bounds__(kSpThreads, 2) skinny_plus_one_kernel(const __grid_constant__ SkinnyPlusArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sm_a = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sm_b = sm_a + kSpABufs * kSpABuf;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm_b + kSpABufs * kSpBBuf);
  __shared__ uint32_t tmem_base_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Codes of both operands ready (16 + 1 warps), a buffer free, a row block's sums ready, drained.
  const uint32_t full = smem_u32(bars), empty = full + 8 * kSpABufs, accf = empty + 8 * kSpABufs, acce = accf + 8,
                 drain_bar = acce + 8;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSpABufs; ++s) {
      mbar_init(full + 8 * s, kSpCodeWarps + 1);
      mbar_init(empty + 8 * s, 1);
    }
    mbar_init(accf, 1);
    mbar_init(acce, kSpCodeWarps);
    mbar_init(drain_bar, 1);
    fence_barrier_init();
  }
  if (warp == kSpCodeWarps) {
    tmem_alloc(smem_u32(&tmem_base_s), 128);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  pdl_wait();  // exponents, flags, the skinny operand's codes, U zero
  const int64_t u0 = a.total * blockIdx.x / gridDim.x, u1 = a.total * (blockIdx.x + 1) / gridDim.x;
  const int64_t first_rb = u0 / a.chunks;
  const int64_t first_chunk = u0 - first_rb * a.chunks;
  const int units = static_cast<int>(u1 - u0);
  bool ok = true;

  if (warp == kSpCodeWarps + 1) {
    // ---------------- B's codes ----------------
    int64_t chunk = first_chunk;
    for (int t = 0; t < units && ok; ++t) {
      const uint32_t s = t % kSpABufs;
      ok = mbar_wait_warp(empty + 8 * s, ((t / kSpABufs) & 1) ^ 1, kWaitLimit);
      if (!ok) break;
      uint8_t* dst = sm_b + s * kSpBBuf;
      const int pieces = a.npad * (kSpK / 16);
      for (int i = lane; i < pieces; i += 32) {  // 16 codes each: column i / 4, K column i mod 4
        const int c = i >> 2, kc = i & 3;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (c < a.cols) v = __ldg(reinterpret_cast<const uint4*>(a.codes + c * a.k_pad + chunk * kSpK + 16 * kc));
        *reinterpret_cast<uint4*>(dst + (kc * a.npad + c) * 16) = v;
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(full + 8 * s);
      if (++chunk == a.chunks) chunk = 0;
    }
    if (!ok && lane == 0) {
      a.dev->status = kStatusTimeout;
      a.dev->timeout_site = 17;
    }
  } else if (warp == kSpCodeWarps) {
    // ---------------- MMA issuer ----------------
    const uint32_t me = lane == 0;
    const uint32_t idesc = idesc_f8_f32(kRows, a.npad);
    const uint64_t da = smem_desc_plain(smem_u32(sm_a), kSpATile, 128);
    const uint64_t db = smem_desc_plain(smem_u32(sm_b), a.npad * 16, 128);
    int64_t chunk = first_chunk;
    uint32_t blocks = 0, fresh = 0;  // row blocks begun; whether the sums hold this one's
    for (int t = 0; t < units && ok; ++t) {
      const uint32_t s = t % kSpABufs;
      if (!fresh) ok = mbar_wait_warp(acce, (blocks & 1) ^ 1, kWaitLimit);
      ok = ok && mbar_wait_warp(full + 8 * s, (t / kSpABufs) & 1, kWaitLimit);
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < kSpK / 32; ++kk)
        mma_f8_by(me, tmem, da + s * (kSpABuf >> 4) + kk * (2 * kSpATile >> 4),
                  db + s * (kSpBBuf >> 4) + kk * (2 * a.npad * 16 >> 4), idesc, kk ? 1u : fresh);
      mma_commit_by(me, empty + 8 * s);
      fresh = 1;
      if (++chunk == a.chunks || t + 1 == units) {
        mma_commit_by(me, accf);
        chunk = 0;
        fresh = 0;
        ++blocks;
      }
    }
    if (!ok && me) {
      a.dev->status = kStatusTimeout;
      a.dev->timeout_site = 18;
    }
    mma_commit_by(me, drain_bar);
    mbar_wait_bounded(drain_bar, 0, kWaitLimit);
    __syncwarp();
  } else {
    // ---------------- A's codes, and the sums ----------------
    const int rq = warp & 3, cq = warp >> 2;
    // 16 entries (`part` of a chunk) of a row.
    const int rloc = 32 * rq + lane, part = cq;
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(32 * rq) << 16);
    int64_t rb = first_rb, chunk = first_chunk;
    const double* p = nullptr;
    int ex = 0;
    bool live = false;
    auto enter = [&]() {
      const int64_t row = rb * kRows + rloc;
      live = row < a.rows && !(a.flag[row] & 2);
      ex = live ? a.scan[row] : 0;
      p = a.A + (row < a.rows ? row : a.rows - 1);
    };
    auto fetch = [&](int64_t c, double (&x)[16]) {
      const int64_t l = c * kSpK + part * 16;
      const double* e = p + l * a.lda;
      if (l + 16 <= a.k) {
#pragma unroll
        for (int j = 0; j < 16; ++j, e += a.lda) x[j] = __ldg(e);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j, e += a.lda) x[j] = l + j < a.k ? __ldg(e) : 0.0;
      }
    };
    enter();
    double x[16];
    fetch(chunk, x);
    uint32_t blocks = 0;
    for (int t = 0; t < units && ok; ++t) {
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t v = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) v |= magnitude_code(x[4 * j + i], ex, a.clamp) << (8 * i);
        w[j] = live ? v : 0u;
      }
      const bool ends = chunk + 1 == a.chunks || t + 1 == units;
      const int64_t out_rb = rb;
      if (t + 1 < units) {
        if (++chunk == a.chunks) {
          chunk = 0;
          ++rb;
          enter();
        }
        fetch(chunk, x);
      }
      const uint32_t s = t % kSpABufs;
      ok = mbar_wait_warp(empty + 8 * s, ((t / kSpABufs) & 1) ^ 1, kWaitLimit);
      if (!ok) break;
      *reinterpret_cast<uint4*>(sm_a + s * kSpABuf + part * kSpATile + rloc * 16) = make_uint4(w[0], w[1], w[2], w[3]);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(full + 8 * s);
      if (ends) {  // the row block's sums (of this run) into U
        ok = mbar_wait_warp(accf, blocks & 1, kWaitLimit);
        if (!ok) break;
        tc_fence_after();
        const int64_t row = out_rb * kRows + 32 * rq + lane;
        for (int c = 4 * cq; c < a.npad; c += 16) {
          uint32_t v[4];
          tmem_ld4(lane_addr + c, v);
          tmem_ld_wait();
          if (row < a.rows) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (c + j < a.cols) atomicAdd(a.U + row * a.ldu + c + j, __uint_as_float(v[j]));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce);
        ++blocks;
      }
    }
    if (!ok && lane == 0) {
      a.dev->status = kStatusTimeout;
      a.dev->timeout_site = 19;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kSpCodeWarps) tmem_dealloc(tmem, 128);
}

static size_t skinny_smem() {
  return 1024 + 2 * static_cast<size_t>(kSnABuf) + kSnBStages * static_cast<size_t>(kSnBChunk) + 8 * (8 + 2 * kSnBStages + 1);
}

struct SkinnyPlan {
  int64_t tall, cols, nrb, groups, slabs, total, grid;
  int slots;
  size_t parts_off, bytes;
};
static SkinnyPlan skinny_plan(int64_t m, int64_t n, int64_t k) {
  SkinnyPlan p;
  p.tall = std::max(m, n);
  p.cols = std::min(m, n);
  p.nrb = (p.tall + kRows - 1) / kRows;
  p.groups = (p.cols + kSnCols - 1) / kSnCols;
  p.slabs = (k + kSnK * kSnSlabChunks - 1) / (kSnK * kSnSlabChunks);
  p.total = p.groups * p.nrb * p.slabs;
  p.grid = std::min<int64_t>(num_sms(), p.total);
  // A run of at least ⌊total/grid⌋ units: a row block's slabs touch at most this many runs.
  p.slots = static_cast<int>((p.slabs + p.total / p.grid - 1) / (p.total / p.grid)) + 1;
  p.parts_off = static_cast<size_t>(p.groups * p.slabs * kSnSlabChunks) * kSnBChunk;
  p.bytes = p.parts_off + static_cast<size_t>(p.groups * p.nrb) * p.slots * kSnWords * kSnOutputs * sizeof(uint32_t);
  return p;
}

// Each 16 rows or columns of C read and convert the tall operand once more,
// 0.77 ms for 16384×16384 entries; the residue path writes and reads its P
// digit planes once, 1.09 + 0.0753·P ms (2.0 at r = 6, P = 12; 3.4 at r = 12,
// P = 30; 4.3 at r = 16, P = 42).  The line is where they meet: 1 to 5 groups
// of 16.  (Measured: 16384×64×16384 r = 12 3.90 ms a call against 4.23, r = 6
// 3.85 against 2.83; 500×64×20000 0.227 against 0.255; 16×16×128 alike.)
bool skinny_applies(int64_t m, int64_t n, int64_t k, int planes, size_t scratch_bytes) {
  return std::min(m, n) <= kSnCols * ((14 + planes) / 10) && skinny_plan(m, n, k).bytes <= scratch_bytes;
}

// Where A is larger than L2; below that the plane stays there and the pass only
// adds a launch (4000×30×4000 alike, 128×48×20000 97 against 126 µs).
bool skinny_plus_one_applies(int64_t m, int64_t n, int64_t k) { return n <= m && m * k >= (int64_t{1} << 24); }

// U = ÂB̂ into the zeroed sums of `split` (m×n row-major, ld n to a multiple of
// 4) and its row maxima.  `codes` are B's magnitude codes.
cudaError_t launch_skinny_plus_one(int64_t m, int64_t n, int64_t k, const double* A, int64_t lda, const int32_t* ra,
                                   const uint8_t* row_flag, const uint8_t* codes, const MagnitudeSplit& split,
                                   float* urow, int* u_max, Oz2Device* dev, cudaStream_t st) {
  SkinnyPlusArgs a{};
  a.A = A;
  a.lda = lda;
  a.rows = m;
  a.k = k;
  a.k_pad = (k + kKPad - 1) / kKPad * kKPad;
  a.nrb = (m + kRows - 1) / kRows;
  a.chunks = a.k_pad / kSpK;
  a.total = a.nrb * a.chunks;
  a.scan = ra;
  a.flag = row_flag;
  a.clamp = magnitude_clamp(k);
  a.codes = codes;
  a.cols = n;
  a.npad = static_cast<int>((n + 15) / 16 * 16);
  a.U = split.sums;
  a.ldu = split.count / m;
  a.dev = dev;
  const void* kern = reinterpret_cast<const void*>(skinny_plus_one_kernel);
  const size_t smem = 1024 + kSpABufs * static_cast<size_t>(kSpABuf + kSpBBuf) + 8 * (2 * kSpABufs + 3);
  cudaError_t err = allow_smem(kern, smem);
  if (err != cudaSuccess) return err;
  count_launch();
  const int64_t grid = std::min<int64_t>(2 * num_sms(), a.total);
  err = launch_dependent(skinny_plus_one_kernel, dim3(static_cast<unsigned>(grid)), dim3(kSpThreads), smem, st, a);
  return err != cudaSuccess ? err : launch_plus_one_rowmax(split.sums, m, n, a.ldu, urow, u_max, st);
}

cudaError_t launch_skinny(int64_t m, int64_t n, int64_t k, const double* A, int64_t lda, const double* B, int64_t ldb,
                          const int32_t* ra, const int32_t* cb, const int32_t* d, const int32_t* e,
                          const uint8_t* row_flag, const uint8_t* col_flag, uint8_t* scratch, double* C, int64_t ldc,
                          Oz2Device* dev, cudaStream_t st) {
  const SkinnyPlan p = skinny_plan(m, n, k);
  const bool b_tall = n > m;
  SkinnyArgs a{};
  a.T = b_tall ? B : A;
  a.row_stride = b_tall ? ldb : 1;
  a.k_stride = b_tall ? 1 : lda;
  a.rows = p.tall;
  a.k = k;
  a.nrb = p.nrb;
  a.slabs = p.slabs;
  a.total = p.total;
  a.exps = b_tall ? e : d;
  a.scan = b_tall ? cb : ra;
  a.flag = b_tall ? col_flag : row_flag;
  a.s_exps = b_tall ? d : e;
  a.s_scan = b_tall ? ra : cb;
  a.s_flag = b_tall ? row_flag : col_flag;
  a.cols = p.cols;
  a.digits = scratch;
  a.parts = reinterpret_cast<uint32_t*>(scratch + p.parts_off);
  a.slots = p.slots;
  a.vec = b_tall && ldb % 2 == 0 && reinterpret_cast<uintptr_t>(B) % 16 == 0;
  a.dev = dev;
  for (int i = 0; i < 4; ++i) a.pow256[i] = 1 << (8 * i);
  const int64_t chunks = p.slabs * kSnSlabChunks;
  const int64_t threads = p.groups * chunks * (kSnK / 8) * kSnCols;
  count_launch(3);
  cudaError_t err =
      launch_dependent(skinny_digits_kernel, dim3(static_cast<unsigned>((threads + 255) / 256)), dim3(256), 0, st,
                       b_tall ? A : B, b_tall ? int64_t{1} : ldb, b_tall ? lda : int64_t{1}, p.cols, k, a.s_exps,
                       a.s_flag, chunks, p.groups, scratch);
  if (err != cudaSuccess) return err;
  const size_t smem = skinny_smem();
  auto kern = b_tall ? skinny_kernel<true> : skinny_kernel<false>;
  err = allow_smem(reinterpret_cast<const void*>(kern), smem);
  if (err != cudaSuccess) return err;
  err = launch_dependent(kern, dim3(static_cast<unsigned>(p.grid)), dim3(kSnThreads), smem, st, a);
  if (err != cudaSuccess) return err;
  return launch_dependent(skinny_finish_kernel, dim3(static_cast<unsigned>(p.groups * p.nrb), kSnCols), dim3(kRows), 0,
                          st, static_cast<const uint32_t*>(a.parts), p.slabs, p.total, p.grid, p.slots, p.nrb, p.tall, p.cols, a.exps,
                          a.s_exps, C, b_tall ? ldc : int64_t{1}, b_tall ? int64_t{1} : ldc);
}

}  // namespace oz2
