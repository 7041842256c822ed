// Phase 2 of Ozaki Scheme II on FP8 tensor cores (§2.3 Eq. modgemm; §2.5
// Eq. sq-shortcut, Eq. kar, Eq. accum-exact) and the "+1" magnitude GEMM of
// §2.4, as one persistent tcgen05 kernel for sm_103a running on CTA pairs.
//
// Work unit = (modulus, 256×256 output tile); units are taken modulus-major
// so that the planes of one modulus stay in L2 while every pair works on it.
// The nonsquare moduli, whose units load three stage pairs per k-block
// against two for a square modulus, come first, and successive waves of
// units are dealt to the pairs in alternating directions, so that the pairs
// that take a heavy unit in one wave take a light one in the next.
// A pair (cluster of 2 CTAs) computes its tile with cta_group::2 MMAs of
// M = N = 256, K = 32: each CTA holds 128 rows of the A plane tile and 128
// rows of the B plane tile in its own shared memory, and 128 rows × 256
// columns of each FP32 accumulator in its tensor memory.
//
// Per modulus the three plane products of §2.5 accumulate into two TMEM
// accumulators (256 columns each):
//   square m = s²  : acc0 += d0·e0,            acc1 += d1·e0 + d0·e1
//   nonsquare m    : acc0 += (d0+d1)(e0+e1),   acc1 += d0·e0 + (-16 d1)·e1
// (the A operand stores its last nonsquare plane pre-scaled by -2^b, the
// accumulator merge of §2.5 "Accumulators").  Every K-slab (32768 squares,
// 4096 nonsquare: Eq. accum-exact) the epilogue reads the accumulators and
// adds  acc0 + s·acc1  or  16·acc0 - 15·acc1  mod m to the residue it keeps
// in registers; after the last slab it stores the centred residue as int16,
// column-major (each thread owns one row; a warp's store covers 32
// consecutive rows of one column, 64 contiguous bytes).
//
// Pipeline: a stage is one (A plane, B plane) pair of 128-byte-deep tiles
// (32 KiB per CTA), six stages.  Warp 0 of each CTA issues its CTA's TMA
// loads, completing on the leader's stage barrier; warp 1 of the leader
// issues the MMAs and multicasts stage releases and accumulator-ready
// signals to both CTAs; warps 2..17 of both CTAs run the epilogue (64
// columns each) and release the accumulators to the leader.  Every wait is
// bounded; on expiry the kernel records OZ2_ERR_TIMEOUT in the device status
// word and drains.
//
// Two kernels share this: residue_gemm_kernel (k > 128), which orders a
// unit's products so that each accumulator is drained while the tensor cores
// work on the other one (and which has a 64-column form for a C of less than
// one wave of those tiles), and plane_gemm_kernel, for the one-k-block residue
// GEMM and the magnitude GEMM, whose units are over before such an overlap
// could start or use one accumulator only.
#include <algorithm>
#include <mutex>
#include <vector>

#include "oz2_gemm.cuh"

namespace oz2 {

constexpr int kTileM = 256, kTileN = 256;        // per CTA pair
constexpr int kStageBytes = 2 * kTileBytes;      // A tile + B tile
constexpr int kStages = 6;
constexpr int kEpiWarps = 16;
constexpr int kGemmThreads = 32 * (2 + kEpiWarps);  // producer, MMA, epilogue
constexpr int kTmemCols = 512;
constexpr int kAccCols = 256;
constexpr int kGroupM = 8;                       // tile rasterisation group

struct EpiCtx {
  int16_t* res;   // r × (m×n column-major, ld = ldr ≥ m; matrix i at i·n·ldr)
  float* urow;
  int* u_max;     // float bits of max_ij U_ij
  Oz2Device* dev;
  int64_t m, n, ldr;
  float* upart;   // magnitude GEMM split along k: U (m×n row-major, ld = ldu) summed over the parts
  int64_t ldu;    // a multiple of 4: 16-byte rows
};

// Units: (modulus, part of the k-blocks, tile).  With kparts > 1 (split K)
// each unit covers kpart_steps consecutive k-blocks (the last part fewer)
// and the epilogue stores its residue as part `part` of the partial-residue
// planes, which fold_parts_kernel then sums mod m (Eq. modgemm is a sum over
// k, so C^(i) is the sum of the parts' residues mod m_i).
struct UnitMap {
  int64_t ntm, ntn, ntiles, nunits;
  int nsq, nheavy;  // leading square moduli; nonsquare moduli after them
  int64_t ksteps, kparts, kpart_steps;
};

struct Unit {
  int i, part;         // modulus, part of the k-blocks
  int64_t tm, tn;      // tile
  int64_t k_lo, k_hi;  // k-blocks [k_lo, k_hi)
};

// Unit u (grouped raster of kGroupM tile rows).  Modulus block j of the
// units is modulus nsq + j for the nheavy nonsquare moduli, then modulus
// j - nheavy for the squares; within a modulus the parts come in order.
// The magnitude GEMM (MODE 1) has one modulus; its parts of k (when it is
// split) come in order, each over all tiles.
template <int MODE>
__device__ __forceinline__ Unit unit_at(int64_t u, const UnitMap& um) {
  Unit x;
  int64_t t = u;
  if (MODE == 1) {
    x.i = 0;
    x.part = static_cast<int>(u / um.ntiles);
    t = u - static_cast<int64_t>(x.part) * um.ntiles;
  } else {
    const int64_t per_mod = um.ntiles * um.kparts;
    const int j = static_cast<int>(u / per_mod);
    x.i = j < um.nheavy ? um.nsq + j : j - um.nheavy;
    const int64_t v = u - static_cast<int64_t>(j) * per_mod;
    x.part = static_cast<int>(v / um.ntiles);
    t = v - static_cast<int64_t>(x.part) * um.ntiles;
  }
  const int64_t per_group = kGroupM * um.ntn;
  const int64_t g = t / per_group;
  const int64_t first = g * kGroupM;
  const int64_t gm = um.ntm - first < kGroupM ? um.ntm - first : kGroupM;
  const int64_t local = t - g * per_group;
  x.tm = first + local % gm;
  x.tn = local / gm;
  x.k_lo = static_cast<int64_t>(x.part) * um.kpart_steps;
  x.k_hi = um.ksteps - x.k_lo < um.kpart_steps ? um.ksteps : x.k_lo + um.kpart_steps;
  return x;
}

// The unit a pair takes in wave w: waves of npairs units, dealt to the pairs
// in ascending order in even waves and descending order in odd ones.
__device__ __forceinline__ int64_t wave_unit(int64_t pair, int64_t w, int64_t npairs) {
  return w * npairs + ((w & 1) ? npairs - 1 - pair : pair);
}

template <int MODE>
__device__ __forceinline__ int planes_of(const Oz2Moduli& mods, int i) {
  return MODE == 0 ? (mods.sq_base[i] ? 2 : 3) : 1;
}
// MODE 0: residue planes (all moduli) for k ≤ 128: one k-block, so one short
// slab for every modulus, whose epilogue takes the single-correction
// reduction.  MODE 1: magnitude planes ("+1" pass); with PARTS its tiles run
// in parts of k and add their partial sums into U (EpiCtx::upart) instead of
// taking row maxima.
template <int MODE, bool PARTS = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
    plane_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                      const __grid_constant__ Oz2Moduli mods, int64_t k_pad, UnitMap um, EpiCtx ctx) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  // bars: full[S], empty[S], acc_full, acc_empty, drain
  __shared__ uint32_t tmem_base_s;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int64_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kStages);
  const uint32_t acc_full = smem_u32(bars + 2 * kStages), acc_empty = smem_u32(bars + 2 * kStages + 1);
  const uint32_t drain_bar = smem_u32(bars + 2 * kStages + 2);
  const int64_t ksteps = k_pad / kBK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 2 * kEpiWarps);
    mbar_init(drain_bar, 1);
    fence_barrier_init();
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmB);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tmem_base_s), kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  bool ok = true;
  pdl_wait();  // the planes are written; the set-up above overlaps that kernel's tail

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs) ----------------
    if (lane == 0) {
      uint32_t it = 0;
      const uint32_t full_leader0 = mapa_shared(full0, 0);
      for (int64_t w = 0, u = pair; u < um.nunits && ok; u = wave_unit(pair, ++w, npairs)) {
        const Unit x = unit_at<MODE>(u, um);
        const int i = x.i;
        const int64_t tm = x.tm, tn = x.tn;
        const int np = planes_of<MODE>(mods, i);
        const int pbase = MODE == 0 ? mods.plane_off[i] : 0;
        const int ya = static_cast<int>(tm * kTileM + rank * kRows);
        const int yb = static_cast<int>(tn * kTileN + rank * kRows);
        // Digit planes: first line of block (row block, k-block 0, plane pbase);
        // successive k-blocks are nplanes blocks apart.  A row block past the
        // operand's last one lies past the end of the tensor (zero fill).
        const int64_t blk_a = (static_cast<int64_t>(ya / kPlaneRows) * ksteps * mods.nplanes + pbase) * kPlaneRows;
        const int64_t blk_b = (static_cast<int64_t>(yb / kPlaneRows) * ksteps * mods.nplanes + pbase) * kPlaneRows;
        for (int64_t kb = x.k_lo; kb < x.k_hi && ok; ++kb) {
          for (int p = 0; p < np; ++p, ++it) {
            const int s = it % kStages;
            if (!mbar_wait_bounded(empty0 + 8 * s, ((it / kStages) & 1) ^ 1, kWaitLimit)) {
              ok = false;
              break;
            }
            if (leader) mbar_arrive_expect_tx(full0 + 8 * s, 2u * kStageBytes);
            const uint32_t sa = smem_u32(smem + s * kStageBytes);
            if (MODE == 0) {
              const int64_t off = (kb * mods.nplanes + p) * kPlaneRows;
              tma_load_2d_pair(sa, &tmA, full_leader0 + 8 * s, 0, static_cast<int>(blk_a + off));
              tma_load_2d_pair(sa + kTileBytes, &tmB, full_leader0 + 8 * s, 0, static_cast<int>(blk_b + off));
            } else {
              const int x = static_cast<int>(kb * kBK);
              tma_load_3d_pair(sa, &tmA, full_leader0 + 8 * s, x, ya, 0);
              tma_load_3d_pair(sa + kTileBytes, &tmB, full_leader0 + 8 * s, x, yb, 0);
            }
          }
        }
      }
      if (!ok) {
        ctx.dev->status = kStatusTimeout;
        ctx.dev->timeout_site = 1;
      }
      if (leader)  // the leader's stage barriers also count the peer's bytes
        for (uint32_t j = (it > kStages ? it - kStages : 0); j < it; ++j)
          mbar_wait_bounded(full0 + 8 * (j % kStages), (j / kStages) & 1, kWaitLimit);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA) ----------------
    if (leader) {  // the whole warp; lane 0 issues
      const uint32_t me = lane == 0;
      constexpr uint32_t idesc = idesc_f8_f32(kTileM, kTileN);
      // Stage s, operand o, k-chunk kk: the descriptor of stage 0 plus the
      // byte offset >> 4 (the start-address field has room: smem < 256 KiB).
      const uint64_t desc0 = smem_desc_sw128(smem_u32(smem));
      uint32_t st = 0, ph = 0, accph = 0;   // current stage and its full-barrier parity
      auto next = [&](uint32_t& s_, uint32_t& p_) {
        if (++s_ == kStages) {
          s_ = 0;
          p_ ^= 1;
        }
      };
      for (int64_t w = 0, u = pair; u < um.nunits && ok; u = wave_unit(pair, ++w, npairs)) {
        const Unit x = unit_at<MODE>(u, um);
        const int i = x.i;
        const int np = planes_of<MODE>(mods, i);
        ok = mbar_wait_warp(acc_empty, accph ^ 1, kWaitLimit);
        if (!ok) break;
        tc_fence_after();
        for (int64_t kb = x.k_lo; kb < x.k_hi && ok; ++kb) {
          const uint32_t first = kb == x.k_lo ? 0u : 1u;
          if (np == 2) {  // square: stages (d0,e0) and (d1,e1)
            uint32_t s1 = st, p1 = ph;
            next(s1, p1);
            ok = mbar_wait_warp(full0 + 8 * st, ph, kWaitLimit) && mbar_wait_warp(full0 + 8 * s1, p1, kWaitLimit);
            if (!ok) break;
            tc_fence_after();
            const uint64_t a0 = desc0 + st * (kStageBytes >> 4), b0 = a0 + (kTileBytes >> 4);
            const uint64_t a1 = desc0 + s1 * (kStageBytes >> 4), b1 = a1 + (kTileBytes >> 4);
#pragma unroll
            for (int kk = 0; kk < kBK / 32; ++kk) {
              const uint32_t acc = kk ? 1u : first;
              mma_f8_pair(me, tmem, a0 + 2 * kk, b0 + 2 * kk, idesc, acc);                 // d0·e0
              mma_f8_pair(me, tmem + kAccCols, a1 + 2 * kk, b0 + 2 * kk, idesc, acc);      // d1·e0
              mma_f8_pair(me, tmem + kAccCols, a0 + 2 * kk, b1 + 2 * kk, idesc, 1u);       // + d0·e1
            }
            mma_commit_pair_mc(me, empty0 + 8 * st, 0x3);
            mma_commit_pair_mc(me, empty0 + 8 * s1, 0x3);
            st = s1;
            ph = p1;
            next(st, ph);
          } else {
            for (int p = 0; p < np; ++p) {  // nonsquare: Σ·Σ → acc0; d0e0, -16 d1·e1 → acc1
              ok = mbar_wait_warp(full0 + 8 * st, ph, kWaitLimit);
              if (!ok) break;
              tc_fence_after();
              const uint32_t col = p == 0 ? 0u : kAccCols;
              const uint64_t a = desc0 + st * (kStageBytes >> 4), b = a + (kTileBytes >> 4);
#pragma unroll
              for (int kk = 0; kk < kBK / 32; ++kk) {
                const uint32_t acc = (kk || p == 2) ? 1u : first;
                mma_f8_pair(me, tmem + col, a + 2 * kk, b + 2 * kk, idesc, acc);
              }
              mma_commit_pair_mc(me, empty0 + 8 * st, 0x3);
              next(st, ph);
            }
          }
        }
        if (!ok) break;
        mma_commit_pair_mc(me, acc_full, 0x3);  // the unit's accumulators complete, both CTAs
        accph ^= 1;
      }
      if (!ok && me) {
        ctx.dev->status = kStatusTimeout;
        ctx.dev->timeout_site = 2;
      }
      // All MMAs retired before the tensor memory or the peer's shared memory goes away.
      mma_commit_pair(me, drain_bar);
      mbar_wait_bounded(drain_bar, 0, kWaitLimit);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue (warps 2..17, both CTAs) ----------------
    const int q = warp & 3;                    // TMEM lane quarter of this warp
    const int h = (warp - 2) >> 2;             // 64-column quarter of the tile
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(32 * q) << 16) + static_cast<uint32_t>(64 * h);
    const uint32_t acc_empty_leader = mapa_shared(acc_empty, 0);
    uint32_t accph = 0;
    for (int64_t w = 0, u = pair; u < um.nunits && ok; u = wave_unit(pair, ++w, npairs)) {
      const Unit x = unit_at<MODE>(u, um);
      const int i = x.i;
      const int64_t tm = x.tm, tn = x.tn;
      const int64_t row = tm * kTileM + rank * kRows + 32 * q + lane;
      const int64_t col0 = tn * kTileN + 64 * h;
      const bool square = MODE == 0 ? mods.sq_base[i] != 0 : true;
      const float mf = MODE == 0 ? static_cast<float>(mods.m[i]) : 1.f;
      const float inv = 1.f / mf;
      const float sb = MODE == 0 ? static_cast<float>(mods.sq_base[i]) : 0.f;
      const float hi = MODE == 0 ? static_cast<float>(mods.m[i] - 1 - mods.m[i] / 2) : 0.f;
      // This thread's row of C^(i); column j at rrow[j·ldr] (a warp stores 32
      // consecutive rows of one column, 64 contiguous bytes, per instruction).
      int16_t* rrow = MODE == 0 ? ctx.res + static_cast<size_t>(i) * ctx.n * ctx.ldr + row : nullptr;
      float rowmax = 0.f;
      if (!mbar_wait_bounded(acc_full, accph, kWaitLimit)) {
        ok = false;
        break;
      }
      tc_fence_after();
#pragma unroll 2
      for (int c = 0; c < 64; c += 16) {
        uint32_t v0[16], v1[16];
        tmem_ld16(lane_addr + c, v0);
        if (MODE == 0) tmem_ld16(lane_addr + kAccCols + c, v1);
        tmem_ld_wait();
        if (c == 48) {
          // The last chunk is in registers: release the accumulators now, so
          // the next unit's MMAs overlap this chunk's reduction and stores.
          // The arrive is relaxed: the residue stores before it need no
          // ordering against the MMAs, and a release would wait for them to
          // be performed.
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote_relaxed(acc_empty_leader);
        }
        if (MODE == 1 && PARTS) {  // a part of k: add this tile's partial sums into U
          const int64_t cc = col0 + c;
          if (row < ctx.m) {
            float* dst = ctx.upart + row * ctx.ldu + cc;  // 16-byte aligned: ldu and cc multiples of 4
            if (cc + 16 <= ctx.n) {
#pragma unroll
              for (int j = 0; j < 16; j += 4)
                atomicAdd(reinterpret_cast<float4*>(dst + j),
                          make_float4(__uint_as_float(v0[j]), __uint_as_float(v0[j + 1]), __uint_as_float(v0[j + 2]),
                                      __uint_as_float(v0[j + 3])));
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (cc + j < ctx.n) atomicAdd(dst + j, __uint_as_float(v0[j]));
            }
          }
        } else if (MODE == 1) {
#pragma unroll
          for (int j = 0; j < 16; ++j) rowmax = fmaxf(rowmax, __uint_as_float(v0[j]));
        } else if (row < ctx.m) {
          const int64_t cc = col0 + c;
          int16_t* dst = rrow + cc * ctx.ldr;
          const int ncol = ctx.n - cc < 16 ? static_cast<int>(ctx.n - cc) : 16;
          if (ncol == 16 && square) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float rj =
                  combine_residue_short1<true>(__uint_as_float(v0[j]), __uint_as_float(v1[j]), sb, mf, inv, hi);
              *dst = static_cast<int16_t>(as_i16_bits(rj));
              dst += ctx.ldr;
            }
          } else if (ncol == 16) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float rj =
                  combine_residue_short1<false>(__uint_as_float(v0[j]), __uint_as_float(v1[j]), sb, mf, inv, hi);
              *dst = static_cast<int16_t>(as_i16_bits(rj));
              dst += ctx.ldr;
            }
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float v = fmaf(square ? 1.f : 16.f, __uint_as_float(v0[j]), (square ? sb : -15.f) * __uint_as_float(v1[j]));
              if (j < ncol) *dst = static_cast<int16_t>(as_i16_bits(short_residue(v, mf, inv, hi)));
              dst += ctx.ldr;
            }
          }
        }
      }
      accph ^= 1;
      if (MODE == 1 && !PARTS) {
        // rows past m hold zeros (TMA fills out-of-range rows with 0)
        if (row < ctx.m) atomicMax(reinterpret_cast<int*>(ctx.urow) + row, __float_as_int(rowmax));
        const int wm = __reduce_max_sync(0xffffffffu, __float_as_int(rowmax));
        if (lane == 0) atomicMax(ctx.u_max, wm);
      }
    }
    if (!ok) {
      ctx.dev->status = kStatusTimeout;
      ctx.dev->timeout_site = 3;
    }
  }
  tc_fence_before();
  cluster_sync_all();  // neither CTA leaves while the pair's MMAs or loads may touch it
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, kTmemCols);
}

// ---------------------------------------------------------------------------
// The residue GEMM for k > 128.
//
// What bounds it: the tensor pipes and the power cap.  A 256×256×4096 unit is
// 49,152 cycles of MMAs on a pair; it takes about 57,000, at the 1.79 to 1.86
// GHz the SMs hold under this load (2.07 GHz idle; the counters of the kernel
// itself: cycles over nanoseconds), with the MMA issuer waiting 6% of them
// for operands and none for the epilogue.
//
// The two 256-column accumulators fill tensor memory, and draining both after
// a unit left the tensor cores idle for about 4 µs of every unit.  Here the
// products of a K-slab are ordered so that each accumulator is complete well
// before, or started well after, the other:
//   nonsquare: phase A  all k-blocks of (d0+d1)(e0+e1)       → acc0
//              phase B  all k-blocks of d0·e0, (-16 d1)·e1    → acc1
//   square:    phase A  d0·e0 of the first kSplitSteps blocks → acc0
//              phase M  every product of the other blocks     → acc0, acc1
//              phase B  d1·e0 + d0·e1 of the first blocks     → acc1
// The epilogue drains acc0 during phase B and acc1 during the next slab's or
// unit's phase A.  FP32 sums of integers below 2^24 do not depend on the
// order.  A square unit loads its first kSplitSteps d0, e0 tiles twice for
// this (it has the loads to spare: two stages per 12 MMAs against three).
// Between the two drains, and from slab to slab, the residue stays in
// registers, two 16-bit values to a word (no write-back to tensor memory).
//
// Measured (both builds in turn on one GB300, GEMM stage): 4096³ r = 12 1.376
// → 1.285 ms, 2500×3001×2047 r = 15 0.459 → 0.402, 2048³ r = 8 0.136 → 0.129,
// 16384³ r = 13 (whole call, power cap) 130.1 → 120.3.  kSplitSteps 4, 5, 8,
// 12 and 20 gave 0.644, 0.641, 0.646, 0.659 and 0.655 ms on squares alone
// (4096³, r = 6): more blocks cover the drain better and load more.  Asking
// L2 for the operand blocks ahead of the loads (eight k-blocks, the pairs
// that share a block taking turns) changed nothing (1.260 against 1.260 ms),
// nor did the tensor core's operand-A collector on the squares' shared d0.
// ---------------------------------------------------------------------------
constexpr int kSplitSteps = 5;       // k-blocks of a square slab whose two accumulators are filled apart

__device__ __forceinline__ int residue_slab_steps(bool square) {
  return (square ? kKSlabSquare : kKSlabMerged) / kBK;
}

// Two residues of magnitude below 2^15 in one word, biased by 2^15.
constexpr float kPackBias = kRoundMagic + 32768.f;
__device__ __forceinline__ uint32_t pack_residues(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo + kPackBias), __float_as_uint(hi + kPackBias), 0x5410);
}
// w·(residue j of the word), exactly: the biased float times w, less the
// biased zero times w, is an integer below 2^20.
__device__ __forceinline__ float unpack_scaled(uint32_t word, int j, float w) {
  return fmaf(w, __uint_as_float(__byte_perm(word, 0x4B40u, j ? 0x5432 : 0x5410)), -w * kPackBias);
}

// TN: columns of a tile.  256, or 64 for a C so small that its 64-column units
// fill no more than one wave of the CTA pairs: a unit's time is then the drain
// of its accumulators, a quarter as long, on four times the pairs.
template <int TN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
    residue_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ Oz2Moduli mods, int64_t k_pad, UnitMap um, EpiCtx ctx) {
  constexpr int kBTile = TN / 2 * kBK;                 // B rows of a CTA
  constexpr int kStage = kTileBytes + kBTile;
  constexpr int kCols = TN / 4;                        // columns of an epilogue warp
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStage);
  // bars: full[S], empty[S], acc_full[2], acc_empty[2], drain
  __shared__ uint32_t tmem_base_s;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int64_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kStages);
  const uint32_t acc_full = smem_u32(bars + 2 * kStages), acc_empty = smem_u32(bars + 2 * kStages + 2);
  const uint32_t drain_bar = smem_u32(bars + 2 * kStages + 4);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(acc_full + 8 * a, 1);
      mbar_init(acc_empty + 8 * a, 2 * kEpiWarps);
    }
    mbar_init(drain_bar, 1);
    fence_barrier_init();
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmB);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tmem_base_s), 2 * TN);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  bool ok = true;
  pdl_wait();  // the planes are written; the set-up above overlaps that kernel's tail

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs) ----------------
    if (lane == 0) {
      const uint32_t full_leader0 = mapa_shared(full0, 0);
      uint32_t it = 0, s = 0, ph = 1;
      auto load = [&](int line_a, int line_b) {
        if (!mbar_wait_bounded(empty0 + 8 * s, ph, kWaitLimit)) {
          ok = false;
          return;
        }
        if (leader) mbar_arrive_expect_tx(full0 + 8 * s, 2u * kStage);
        const uint32_t sa = smem_u32(smem + s * kStage);
        tma_load_2d_pair(sa, &tmA, full_leader0 + 8 * s, 0, line_a);
        tma_load_2d_pair(sa + kTileBytes, &tmB, full_leader0 + 8 * s, 0, line_b);
        ++it;
        if (++s == kStages) {
          s = 0;
          ph ^= 1;
        }
      };
      const int kb_lines = mods.nplanes * kPlaneRows;  // lines from one k-block's blocks to the next's
      for (int64_t w = 0, u = pair; u < um.nunits && ok; u = wave_unit(pair, ++w, npairs)) {
        const Unit x = unit_at<0>(u, um);
        const bool square = mods.sq_base[x.i] != 0;
        const int slab = residue_slab_steps(square), khi = static_cast<int>(x.k_hi);
        // First lines of this modulus's plane 0 in k-block 0 of the unit's row
        // blocks.  A row block past the operand's last one lies past the end
        // of the tensor (zero fill).
        const int pline = mods.plane_off[x.i] * kPlaneRows;
        const int line_a = static_cast<int>((x.tm * 2 + rank) * um.ksteps * kb_lines) + pline;
        const int row_b = static_cast<int>(x.tn) * TN + static_cast<int>(rank) * (TN / 2);
        const int line_b = static_cast<int>(static_cast<int64_t>(row_b / kPlaneRows) * um.ksteps * kb_lines) + pline +
                           row_b % kPlaneRows;
        auto blocks = [&](int kb0, int kb1, int p0, int np) {
          for (int kb = kb0; kb < kb1 && ok; ++kb) {
            const int off = kb * kb_lines + p0 * kPlaneRows;
            for (int p = 0; p < np && ok; ++p) load(line_a + off + p * kPlaneRows, line_b + off + p * kPlaneRows);
          }
        };
        for (int k0 = static_cast<int>(x.k_lo); k0 < khi && ok; k0 += slab) {
          const int k1 = min(k0 + slab, khi), ke = square ? min(k0 + kSplitSteps, k1) : k1;
          blocks(k0, ke, 0, 1);
          blocks(ke, k1, 0, 2);
          blocks(k0, ke, square ? 0 : 1, 2);
        }
      }
      if (!ok) {
        ctx.dev->status = kStatusTimeout;
        ctx.dev->timeout_site = 1;
      }
      if (leader)  // the leader's stage barriers also count the peer's bytes
        for (uint32_t j = (it > kStages ? it - kStages : 0); j < it; ++j)
          mbar_wait_bounded(full0 + 8 * (j % kStages), (j / kStages) & 1, kWaitLimit);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA) ----------------
    if (leader) {  // the whole warp; lane 0 issues
      const uint32_t me = lane == 0;
      constexpr uint32_t idesc = idesc_f8_f32(kTileM, TN);
      // Stage s, operand o, k-chunk kk: the descriptor of stage 0 plus the
      // byte offset >> 4 (the start-address field has room: smem < 256 KiB).
      const uint64_t desc0 = smem_desc_sw128(smem_u32(smem));
      uint32_t st = 0, ph = 0, accph = 1;  // current stage and its full-barrier parity
      auto wait_stage = [&]() { return ok = mbar_wait_warp(full0 + 8 * st, ph, kWaitLimit); };
      auto release_stage = [&](uint32_t s) { mma_commit_pair_mc(me, empty0 + 8 * s, 0x3); };
      auto next = [&]() {
        if (++st == kStages) {
          st = 0;
          ph ^= 1;
        }
      };
      // One stage into one accumulator.
      auto single = [&](uint32_t col, uint32_t acc) {
        if (!wait_stage()) return;
        tc_fence_after();
        const uint64_t a = desc0 + st * (kStage >> 4), b = a + (kTileBytes >> 4);
#pragma unroll
        for (int kk = 0; kk < kBK / 32; ++kk) mma_f8_pair(me, tmem + col, a + 2 * kk, b + 2 * kk, idesc, kk ? 1u : acc);
        release_stage(st);
        next();
      };
      // A square's stage pair (d0, e0), (d1, e1): d1·e0 + d0·e1 into acc1,
      // and, when `both`, d0·e0 into acc0.
      auto cross = [&](bool both, uint32_t acc0, uint32_t acc1) {
        if (!wait_stage()) return;
        const uint32_t s0 = st;
        next();
        if (!wait_stage()) return;
        const uint32_t s1 = st;
        next();
        tc_fence_after();
        const uint64_t a0 = desc0 + s0 * (kStage >> 4), b0 = a0 + (kTileBytes >> 4);
        const uint64_t a1 = desc0 + s1 * (kStage >> 4), b1 = a1 + (kTileBytes >> 4);
#pragma unroll
        for (int kk = 0; kk < kBK / 32; ++kk) {
          if (both) mma_f8_pair(me, tmem, a0 + 2 * kk, b0 + 2 * kk, idesc, kk ? 1u : acc0);
          mma_f8_pair(me, tmem + TN, a1 + 2 * kk, b0 + 2 * kk, idesc, kk ? 1u : acc1);
          mma_f8_pair(me, tmem + TN, a0 + 2 * kk, b1 + 2 * kk, idesc, 1u);
        }
        release_stage(s0);
        release_stage(s1);
      };
      for (int64_t w = 0, u = pair; u < um.nunits && ok; u = wave_unit(pair, ++w, npairs)) {
        const Unit x = unit_at<0>(u, um);
        const bool square = mods.sq_base[x.i] != 0;
        const int slab = residue_slab_steps(square), khi = static_cast<int>(x.k_hi);
        for (int k0 = static_cast<int>(x.k_lo); k0 < khi && ok; k0 += slab) {
          const int k1 = min(k0 + slab, khi), ke = square ? min(k0 + kSplitSteps, k1) : k1;
          ok = mbar_wait_warp(acc_empty, accph, kWaitLimit);
          tc_fence_after();
          for (int kb = k0; kb < ke && ok; ++kb) single(0, kb != k0);  // phase A
          ok = ok && mbar_wait_warp(acc_empty + 8, accph, kWaitLimit);
          tc_fence_after();
          for (int kb = ke; kb < k1 && ok; ++kb) cross(true, 1u, kb != ke);  // phase M
          if (!ok) break;
          mma_commit_pair_mc(me, acc_full, 0x3);  // acc0 complete for this slab, both CTAs
          if (square) {                       // phase B
            for (int kb = k0; kb < ke && ok; ++kb) cross(false, 1u, ke < k1 || kb != k0);
          } else {
            for (int kb = k0; kb < ke && ok; ++kb) {
              single(TN, kb != k0);
              if (ok) single(TN, 1u);
            }
          }
          if (!ok) break;
          mma_commit_pair_mc(me, acc_full + 8, 0x3);
          accph ^= 1;
        }
      }
      if (!ok && me) {
        ctx.dev->status = kStatusTimeout;
        ctx.dev->timeout_site = 2;
      }
      // All MMAs retired before the tensor memory or the peer's shared memory goes away.
      mma_commit_pair(me, drain_bar);
      mbar_wait_bounded(drain_bar, 0, kWaitLimit);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue (warps 2..17, both CTAs) ----------------
    const int q = warp & 3;                    // TMEM lane quarter of this warp
    const int h = (warp - 2) >> 2;             // column quarter of the tile
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(32 * q) << 16) + static_cast<uint32_t>(kCols * h);
    const uint32_t acc_empty_leader = mapa_shared(acc_empty, 0);
    uint32_t accph = 0;
    uint32_t pk[kCols / 2];  // this thread's running residues, two to a word
    // Columns [c, c + 16) of accumulator a; after the last ones the
    // accumulator is free.  The arrive is relaxed: a release would hold it
    // until the residue stores before it are performed, and the MMAs need no
    // ordering against those.
    auto load16 = [&](int a, int c, uint32_t (&v)[16]) {
      tmem_ld16(lane_addr + a * TN + c, v);
      tmem_ld_wait();
      if (c == kCols - 16) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote_relaxed(acc_empty_leader + 8 * a);
      }
    };
    for (int64_t w = 0, u = pair; u < um.nunits && ok; u = wave_unit(pair, ++w, npairs)) {
      const Unit x = unit_at<0>(u, um);
      const int i = x.i;
      const int64_t row = x.tm * kTileM + rank * kRows + 32 * q + lane;
      const int64_t col0 = x.tn * TN + kCols * h;
      const bool square = mods.sq_base[i] != 0;
      const float mf = static_cast<float>(mods.m[i]);
      const float inv = 1.f / mf;
      const float hi = static_cast<float>(mods.m[i] - 1 - mods.m[i] / 2);
      // v = w0·acc0 + w1·acc1: acc0 + s·acc1 (Eq. sq-shortcut) or
      // 16·acc0 - 15·acc1 (Eq. kar with the merged accumulator).
      const float w0 = square ? 1.f : 16.f, w1 = square ? static_cast<float>(mods.sq_base[i]) : -15.f;
      // This thread's row of C^(i) (of part `part` of it under split K);
      // column j at rrow[j·ldr].
      int16_t* rrow = ctx.res + (static_cast<size_t>(x.part) * mods.r + i) * ctx.n * ctx.ldr + row;
      const int slab = residue_slab_steps(square), khi = static_cast<int>(x.k_hi);
      for (int k0 = static_cast<int>(x.k_lo); k0 < khi; k0 += slab) {
        const bool first = k0 == static_cast<int>(x.k_lo), last = k0 + slab >= khi;
        // acc0, during phase B.  The first slab keeps a = acc0 mod m itself
        // (|a| < 1.5m); a later one adds w0·a to the running residue
        // (|w0·a| + m/2 < 2^14.1) and keeps that within 1.5m.
        if (!mbar_wait_bounded(acc_full, accph, kWaitLimit)) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < kCols; c += 16) {
          uint32_t v[16];
          load16(0, c, v);
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            float a[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              a[t] = loose_mod(__uint_as_float(v[j + t]), mf, inv);
              if (!first) a[t] = loose_mod(fmaf(w0, a[t], unpack_scaled(pk[(c + j) / 2], t, 1.f)), mf, inv);
            }
            pk[(c + j) / 2] = pack_residues(a[0], a[1]);
          }
        }
        // acc1, during the next slab's or unit's phase A.  |v| ≤ 1.5m·(w0 +
        // |w1|) < 2^16 (34·1.5·1089 for squares, 31·1.5·511 otherwise).
        if (!mbar_wait_bounded(acc_full + 8, accph, kWaitLimit)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const float wp = first ? w0 : 1.f;
#pragma unroll
        for (int c = 0; c < kCols; c += 16) {
          uint32_t v[16];
          load16(1, c, v);
          const int64_t cc = col0 + c;
          const int ncol = ctx.n - cc < 16 ? static_cast<int>(ctx.n - cc) : 16;
          auto reduce = [&](int j) {
            const float b = loose_mod(__uint_as_float(v[j]), mf, inv);
            return centred_small(fmaf(w1, b, unpack_scaled(pk[(c + j) / 2], j & 1, wp)), mf, inv, hi);
          };
          if (!last) {
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
              const float r0 = reduce(j), r1 = reduce(j + 1);
              pk[(c + j) / 2] = pack_residues(r0, r1);
            }
          } else if (row < ctx.m) {
            int16_t* dst = rrow + cc * ctx.ldr;
            if (ncol == 16) {
#pragma unroll
              for (int j = 0; j < 16; ++j, dst += ctx.ldr) *dst = static_cast<int16_t>(as_i16_bits(reduce(j)));
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j, dst += ctx.ldr)
                if (j < ncol) *dst = static_cast<int16_t>(as_i16_bits(reduce(j)));
            }
          }
        }
        accph ^= 1;
      }
    }
    if (!ok) {
      ctx.dev->status = kStatusTimeout;
      ctx.dev->timeout_site = 3;
    }
  }
  tc_fence_before();
  cluster_sync_all();  // neither CTA leaves while the pair's MMAs or loads may touch it
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, 2 * TN);
}

// ---------------------------------------------------------------------------
// Tensor-pipe rate probe.  Every CTA pair issues `iters` MMAs of the residue
// GEMM's own form (cta_group::2, kind::f8f6f4, M = N = 256, K = 32) on one
// zero-filled operand tile pair in shared memory, into one accumulator, with
// no loads and no epilogue.  Timed by the caller, it gives the dense FP8 rate
// of the tensor pipes at the clock they run at: the ceiling for the residue
// GEMM, which issues the same instruction.  The shared-memory request keeps
// one CTA per SM, as in the GEMM.
// ---------------------------------------------------------------------------
constexpr int kProbeThreads = 64;
constexpr size_t kProbeSmem = 1024 + 2 * kTileBytes + 64 + 128 * 1024;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kProbeThreads, 1)
    mma_rate_kernel(int64_t iters, Oz2Device* dev) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + 2 * kTileBytes);
  __shared__ uint32_t tmem_base_s;
  const int warp = threadIdx.x >> 5;
  const bool leader = cluster_ctarank() == 0;
  for (int i = threadIdx.x; i < 2 * kTileBytes / 16; i += kProbeThreads)
    reinterpret_cast<uint4*>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async_smem();  // the tensor core reads what the threads wrote
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(bar), 1);
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tmem_base_s), kAccCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  if (leader && warp == 1) {  // the whole warp; lane 0 issues
    const uint32_t me = threadIdx.x == 32;
    constexpr uint32_t idesc = idesc_f8_f32(kTileM, kTileN);
    const uint64_t a = smem_desc_sw128(smem_u32(smem)), b = a + (kTileBytes >> 4);
    for (int64_t it = 0; it < iters; ++it) {
      const uint32_t kk = static_cast<uint32_t>(it & 3);
      mma_f8_pair(me, tmem, a + 2 * kk, b + 2 * kk, idesc, it ? 1u : 0u);
    }
    mma_commit_pair(me, smem_u32(bar));
    if (!mbar_wait_warp(smem_u32(bar), 0, kWaitLimit) && me) {
      dev->status = kStatusTimeout;
      dev->timeout_site = 4;
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();  // the pair's MMAs read both CTAs' shared memory
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, kAccCols);
}

cudaError_t launch_mma_rate(int64_t iters, Oz2Device* dev, int* pairs_out, cudaStream_t st);

// ---------------------------------------------------------------------------
// Plain CUDA-core kernel with the same semantics (diagnostic reference for
// the tensor-core path; accumulates the same integer plane products in FP32
// in sequential k order, so exactness follows from the same bound).
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void plane_gemm_simt_kernel(const uint8_t* __restrict__ pa, const uint8_t* __restrict__ pb,
                                       const __grid_constant__ Oz2Moduli mods, int64_t k_pad, EpiCtx ctx) {
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t col = blockIdx.y;
  if (row >= ctx.m || col >= ctx.n) return;
  const uint8_t* ar = pa + row * k_pad;
  const uint8_t* bc = pb + col * k_pad;
  if (MODE == 1) {  // magnitude planes: one plane, rows × k_pad
    float acc = 0.f;
    for (int64_t l = 0; l < k_pad; ++l) acc += e4m3_to_float(ar[l]) * e4m3_to_float(bc[l]);
    atomicMax(reinterpret_cast<int*>(ctx.urow) + row, __float_as_int(acc));
    atomicMax(ctx.u_max, __float_as_int(acc));
    return;
  }
  for (int i = 0; i < mods.r; ++i) {
    const bool square = mods.sq_base[i] != 0;
    const float mf = static_cast<float>(mods.m[i]);
    const float inv = 1.f / mf;
    const float hi = static_cast<float>(mods.m[i] - 1 - mods.m[i] / 2);
    const int64_t slab = square ? kKSlabSquare : kKSlabMerged;
    // Byte l of plane plane_off + j of row `rw` (of A) or column (of B), in
    // 128 × 128-byte blocks.
    const int64_t kblocks = k_pad / kPlaneLine;
    auto plane = [&](const uint8_t* base, int64_t rw, int j, int64_t l) {
      const int64_t blk = ((rw / kPlaneRows) * kblocks + l / kPlaneLine) * mods.nplanes + mods.plane_off[i] + j;
      return e4m3_to_float(base[blk * kPlaneBlock + (rw % kPlaneRows) * kPlaneLine + l % kPlaneLine]);
    };
    float res = 0.f;
    for (int64_t l0 = 0; l0 < k_pad; l0 += slab) {
      float a0 = 0.f, a1 = 0.f;
      const int64_t l1 = min(k_pad, l0 + slab);
      for (int64_t l = l0; l < l1; ++l) {
        const float x0 = plane(pa, row, 0, l), y0 = plane(pb, col, 0, l);
        const float x1 = plane(pa, row, 1, l), y1 = plane(pb, col, 1, l);
        if (square) {
          a0 += x0 * y0;
          a1 += x1 * y0 + x0 * y1;
        } else {
          const float x2 = plane(pa, row, 2, l), y2 = plane(pb, col, 2, l);
          a0 += x0 * y0;
          a1 += x1 * y1 + x2 * y2;
        }
      }
      res = combine_residue(a0, a1, square, static_cast<float>(mods.sq_base[i]), mf, inv, hi, res);
    }
    ctx.res[static_cast<size_t>(i) * ctx.n * ctx.ldr + col * ctx.ldr + row] = static_cast<int16_t>(res);
  }
}

// ---------------------------------------------------------------------------
// Host side: tensor maps and launch.
// ---------------------------------------------------------------------------
// Magnitude plane of one operand: rows × k_pad bytes, row-major; the box is
// 128 rows × 128 bytes with the 128-byte swizzle the MMA descriptors use.
static bool make_plane_map(CUtensorMap* map, const uint8_t* base, int64_t rows, int64_t k_pad) {
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) return false;
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(k_pad), static_cast<cuuint64_t>(rows), 1};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(k_pad), static_cast<cuuint64_t>(rows * k_pad)};
  cuuint32_t box[3] = {kBK, static_cast<cuuint32_t>(kRows), 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// ---------------------------------------------------------------------------
// Split K.  A problem whose units fill few waves of the CTA pairs (a small C
// with a long k) runs each unit's k-blocks in kparts parts; the parts'
// residues land in scratch planes [part][modulus][column][row] and
// fold_parts_kernel sums them mod m into C^(i).
// ---------------------------------------------------------------------------
constexpr int kFoldThreads = 128;

// C^(i) from its parts: the sum of kparts centred residues has magnitude at
// most kparts·⌊m/2⌋ < 2^16, so centred_small reduces it exactly.  One thread
// takes 8 consecutive rows of one column (16-byte loads: ldr is a multiple
// of 8 and both buffers are 16-byte aligned); blockIdx.z is the modulus.
__global__ void __launch_bounds__(kFoldThreads) fold_parts_kernel(const int16_t* __restrict__ part,
                                                                  int16_t* __restrict__ res, int64_t m, int64_t n,
                                                                  int64_t ldr, int kparts,
                                                                  const __grid_constant__ Oz2Moduli mods) {
  pdl_wait();
  const int i = blockIdx.z;
  const float mf = static_cast<float>(mods.m[i]), inv = 1.f / mf;
  const float hi = static_cast<float>(mods.m[i] - 1 - mods.m[i] / 2);
  const int64_t row0 = (static_cast<int64_t>(blockIdx.x) * kFoldThreads + threadIdx.x) * 8;
  if (row0 >= m) return;
  const size_t plane = static_cast<size_t>(n) * ldr, pstride = static_cast<size_t>(mods.r) * plane;
  for (int64_t col = blockIdx.y; col < n; col += gridDim.y) {
    const size_t off = static_cast<size_t>(i) * plane + static_cast<size_t>(col) * ldr + row0;
    if (row0 + 8 <= m) {
      int acc[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = 0;
      for (int p = 0; p < kparts; ++p) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(part + p * pstride + off));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[2 * j] += static_cast<int16_t>(w[j] & 0xFFFFu);
          acc[2 * j + 1] += static_cast<int>(w[j]) >> 16;
        }
      }
      uint32_t o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        o[j] = as_i16_bits(centred_small(static_cast<float>(acc[2 * j]), mf, inv, hi)) |
               (as_i16_bits(centred_small(static_cast<float>(acc[2 * j + 1]), mf, inv, hi)) << 16);
      *reinterpret_cast<uint4*>(res + off) = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
      for (int64_t r = row0; r < m; ++r) {
        int a = 0;
        for (int p = 0; p < kparts; ++p) a += part[p * pstride + off + (r - row0)];
        res[off + (r - row0)] = static_cast<int16_t>(as_i16_bits(centred_small(static_cast<float>(a), mf, inv, hi)));
      }
    }
  }
}

// At most 16 parts of k.  The fold's sum of kparts centred residues stays
// far inside 16 bits (16·⌊m/2⌋ ≤ 8704); what limits a split in practice is
// the scratch (the magnitude-plane region must hold kparts partial residue
// sets) and the cost model's 5% gain rule.
constexpr int64_t kMaxKParts = 16;
constexpr int64_t kMinPartSteps = 4;   // k-blocks (512 k-entries) per part at least

// Estimated duration of the residue GEMM under the unit schedule (nonsquare
// moduli first, waves dealt in alternating directions), in units of one
// stage pair on a CTA pair (a 256×256×128 FP8 product, about 0.39 µs at
// 2.07 GHz): the largest load over the pairs.  A nonsquare unit of s
// k-blocks costs 3s plus 10 per epilogue drain (one per 4096 k-entries), a
// square one 2s plus 10 per 32768.  A split adds the fold (its bytes at
// about 5 TB/s, and a launch).  The pairs' loads are piecewise constant in
// the pair index, changing only where the heavy units and all units end in
// their last waves, so those pairs and the two ends cover the maximum.
// This is the model that oz2_plan reports and that oz2_dgemm_ex's workspace
// and its callers' saved plans follow; residue_gemm_kernel itself now hides
// most of a drain and takes the same time for either kind of modulus, which
// fastest_kparts below goes by.
static double split_cost(int64_t ntiles, int r, int nsq, int64_t ksteps, int64_t kparts, int64_t pairs, int64_t m,
                         int64_t n) {
  const int64_t s = (ksteps + kparts - 1) / kparts;
  const int64_t U = ntiles * r * kparts, H = ntiles * (r - nsq) * kparts;
  const int64_t P = std::max<int64_t>(1, std::min(pairs, U));
  constexpr int64_t kSlabM = kKSlabMerged / kBK, kSlabS = kKSlabSquare / kBK;
  const double wh = 3.0 * s + 10.0 * ((s + kSlabM - 1) / kSlabM);
  const double wl = 2.0 * s + 10.0 * ((s + kSlabS - 1) / kSlabS);
  auto count = [&](int64_t X, int64_t q) {  // units below X that pair q takes
    const int64_t w0 = X / P, rem = X - w0 * P;
    const int64_t pos = (w0 & 1) ? P - 1 - q : q;
    return w0 + (pos < rem ? 1 : 0);
  };
  auto load = [&](int64_t q) {
    const int64_t h = count(H, q);
    return h * wh + (count(U, q) - h) * wl;
  };
  double mx = std::max(load(0), load(P - 1));
  for (const int64_t X : {H, U}) {
    const int64_t w0 = X / P, rem = X - w0 * P;
    const int64_t b = (w0 & 1) ? P - rem : rem;
    for (const int64_t q : {b - 1, b})
      if (q >= 0 && q < P) mx = std::max(mx, load(q));
  }
  if (kparts > 1) mx += (3.0 + (kparts + 1.0) * r * m * n * 2.0 / 5.0e6) / 0.39;
  return mx;
}

// Parts of K per residue-GEMM unit: 1 unless the units fill fewer than four
// waves and a split of at most max_parts (each part non-empty and at least
// kMinPartSteps k-blocks) is estimated at least 5% faster.
static int64_t choose_kparts(int64_t ntiles, int r, int nsq, int64_t ksteps, int64_t pairs, int64_t m, int64_t n,
                             int64_t max_parts) {
  if (max_parts < 2 || ntiles * r >= 4 * pairs) return 1;
  int64_t best = 1;
  double best_cost = split_cost(ntiles, r, nsq, ksteps, 1, pairs, m, n);
  for (int64_t p = 2; p <= max_parts; ++p) {
    const int64_t s = (ksteps + p - 1) / p;
    if (s < kMinPartSteps) break;
    if ((ksteps + s - 1) / s != p) continue;  // a part would be empty
    const double c = split_cost(ntiles, r, nsq, ksteps, p, pairs, m, n);
    if (c < 0.95 * best_cost) {
      best = p;
      best_cost = c;
    }
  }
  return best;
}

int64_t residue_gemm_kparts(int64_t m, int64_t n, int64_t k_pad, int r, int nsq, int64_t ldr, size_t partial_bytes,
                            int64_t pairs) {
  if (m <= 0 || n <= 0 || k_pad <= 0 || r < 1 || ldr < m || ldr % 8 != 0 || pairs < 1) return 1;
  const size_t part_bytes = static_cast<size_t>(r) * n * ldr * sizeof(int16_t);
  const int64_t max_parts = std::min<int64_t>(kMaxKParts, static_cast<int64_t>(partial_bytes / part_bytes));
  const int64_t ntiles = ((m + kTileM - 1) / kTileM) * ((n + kTileN - 1) / kTileN);
  return choose_kparts(ntiles, r, nsq, k_pad / kBK, pairs, m, n, max_parts);
}

// The parts oz2_dgemm takes, whose plan nobody reads: the fastest by an
// estimate of this kernel, where a unit's time is its k-blocks (0.96 µs each,
// every modulus alike) and about three more, and the fold moves the partial
// residues at 5 TB/s; no split for less than a twentieth.  (1024²×65536, r =
// 12: 192 units of 512 k-blocks in three waves or 960 of 103 in thirteen:
// 2.77 and 2.70 ms a call, both in turn; 900×800×40000 r = 10 1.41 and 1.36,
// 1040×651×47202 r = 8 1.38 and 1.31.)
static int64_t fastest_kparts(int64_t ntiles, int r, int64_t ksteps, int64_t pairs, int64_t m, int64_t n,
                              int64_t max_parts) {
  constexpr double kBlock = 0.96, kUnit = 3.0;  // µs per k-block; a unit's overhead in k-blocks
  int64_t best = 1;
  double best_cost = 1e300;
  for (int64_t p = 1; p <= std::max<int64_t>(1, max_parts); ++p) {
    const int64_t s = (ksteps + p - 1) / p;
    if (p > 1 && (s < kMinPartSteps || (ksteps + s - 1) / s != p)) continue;
    const int64_t waves = (ntiles * r * p + pairs - 1) / pairs;
    double c = static_cast<double>(waves) * (static_cast<double>(s) + kUnit) * kBlock;
    if (p > 1) c += 3.0 + (static_cast<double>(p) + 1.0) * r * static_cast<double>(m) * static_cast<double>(n) * 2.0 / 5.0e6;
    if (c < (best == 1 ? 0.95 : 1.0) * best_cost) {
      best = p;
      best_cost = c;
    }
  }
  return best;
}

static size_t gemm_smem_bytes() { return 1024 + static_cast<size_t>(kStages) * kStageBytes + 8 * (2 * kStages + 5); }

// The magnitude GEMM split along k: each part adds its tiles' partial sums
// into U with 16-byte vector atomics (every partial sum is an integer number
// of units 2^-2c below 2^24, like the whole sum, so FP32 adds them exactly in
// any order), and this kernel then takes each row's maximum, as the unsplit
// epilogue does: a warp per row of the row-major U.
constexpr int kRowMaxThreads = 256;
__global__ void __launch_bounds__(kRowMaxThreads) plus_one_rowmax_kernel(const float* __restrict__ U, int64_t m,
                                                                         int64_t n, int64_t ldu,
                                                                         float* __restrict__ urow, int* u_max) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int64_t row = static_cast<int64_t>(blockIdx.x) * (kRowMaxThreads / 32) + (threadIdx.x >> 5);
  if (row >= m) return;  // whole warps
  float mx = 0.f;
  const float* p = U + row * ldu;
  for (int64_t col = lane; col < n; col += 32) mx = fmaxf(mx, __ldg(p + col));
  const int wm = __reduce_max_sync(0xffffffffu, __float_as_int(mx));  // nonnegative floats order as their bits
  if (lane == 0) {
    atomicMax(reinterpret_cast<int*>(urow) + row, wm);
    atomicMax(u_max, wm);
  }
}

cudaError_t launch_plus_one_rowmax(const float* U, int64_t m, int64_t n, int64_t ldu, float* urow, int* u_max,
                                   cudaStream_t st) {
  constexpr int64_t rows_per_block = kRowMaxThreads / 32;
  count_launch();
  return launch_dependent(plus_one_rowmax_kernel, dim3(static_cast<unsigned>((m + rows_per_block - 1) / rows_per_block)),
                          dim3(kRowMaxThreads), 0, st, U, m, n, ldu, urow, u_max);
}

// The sums of a magnitude GEMM that adds into U anyway (k_skinny.cu).
MagnitudeSplit magnitude_sums(int64_t m, int64_t n, void* scratch) {
  return MagnitudeSplit{2, static_cast<float*>(scratch), m * ((n + 3) / 4 * 4)};
}

// Parts of k for the magnitude GEMM: its 256×256 tiles fill fewer than half
// a wave of the CTA pairs only for a small C with a long k; then each tile
// runs in as many parts as the pairs allow (at most 64, each at least
// kMinPartSteps k-blocks), and U's partial sums go through scratch.
static int64_t magnitude_ldu(int64_t n) { return (n + 3) / 4 * 4; }

static int64_t magnitude_kparts(int64_t ntiles, int64_t ksteps, int64_t pairs, int64_t m, int64_t n,
                                size_t scratch_bytes) {
  if (2 * ntiles >= pairs || scratch_bytes < static_cast<size_t>(m) * magnitude_ldu(n) * sizeof(float)) return 1;
  int64_t p = std::min<int64_t>({64, pairs / ntiles, ksteps / kMinPartSteps});
  if (p < 2) return 1;
  const int64_t s = (ksteps + p - 1) / p;
  return (ksteps + s - 1) / s;  // no empty part
}

int64_t magnitude_gemm_kparts(int64_t m, int64_t n, int64_t k_pad, size_t scratch_bytes, int64_t pairs) {
  if (m <= 0 || n <= 0 || k_pad <= 0 || pairs < 1) return 1;
  const int64_t ntiles = ((m + kTileM - 1) / kTileM) * ((n + kTileN - 1) / kTileN);
  return magnitude_kparts(ntiles, k_pad / kBK, pairs, m, n, scratch_bytes);
}

// A split costs the sums' zeroing, atomics and a launch for the row maxima,
// about 10 µs; a k-block is 0.27 µs of a tile.  With `only_if_faster` a split
// that saves fewer than 36 k-blocks is not made (1000×777×1333: 133 µs a call
// split, 121 unsplit; 1000×1000×8000, 63 k-blocks in 4 parts: 413 and 411;
// 1024×1024×65536: 2830 and 2916).
MagnitudeSplit magnitude_split(int64_t m, int64_t n, int64_t k_pad, void* scratch, size_t scratch_bytes,
                               bool only_if_faster) {
  MagnitudeSplit sp{1, nullptr, 0};
  if (!scratch || reinterpret_cast<uintptr_t>(scratch) % 16 != 0) return sp;
  const void* kern = reinterpret_cast<const void*>(plane_gemm_kernel<1>);
  if (allow_smem(kern, gemm_smem_bytes()) != cudaSuccess) return sp;
  const int64_t p =
      magnitude_gemm_kparts(m, n, k_pad, scratch_bytes, resident_pairs(kern, kGemmThreads, gemm_smem_bytes()));
  const int64_t ksteps = k_pad / kBK;
  if (p < 2 || (only_if_faster && ksteps - (ksteps + p - 1) / p < 36)) return sp;
  sp.parts = p;
  sp.sums = static_cast<float*>(scratch);
  sp.count = m * magnitude_ldu(n);
  return sp;
}

// ---------------------------------------------------------------------------
// Device and kernel facts, kept per (kernel, device).  A device's SM count and
// a kernel's resident clusters on it do not change while a process runs.
// ---------------------------------------------------------------------------
namespace {
struct KernelFact {
  const void* kernel;
  int dev;
  size_t smem;       // dynamic shared memory allowed so far
  int64_t pairs;     // resident two-CTA clusters (0: not asked yet)
};
std::mutex g_fact_mu;
std::vector<KernelFact> g_facts;
int g_sms[64];

int current_device() {
  int dev = 0;
  cudaGetDevice(&dev);
  return dev;
}
KernelFact& fact_of(const void* kernel, int dev) {  // with g_fact_mu held
  for (KernelFact& f : g_facts)
    if (f.kernel == kernel && f.dev == dev) return f;
  g_facts.push_back(KernelFact{kernel, dev, 0, 0});
  return g_facts.back();
}
}  // namespace

int num_sms() {
  const int dev = current_device();
  if (dev < 0 || dev >= 64) return 148;
  std::lock_guard<std::mutex> lk(g_fact_mu);
  if (!g_sms[dev]) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 148;
    g_sms[dev] = sms;
  }
  return g_sms[dev];
}

cudaError_t allow_smem(const void* kernel, size_t smem) {
  const int dev = current_device();
  std::lock_guard<std::mutex> lk(g_fact_mu);
  KernelFact& f = fact_of(kernel, dev);
  if (f.smem >= smem) return cudaSuccess;
  const cudaError_t err =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (err == cudaSuccess) f.smem = smem;
  return err;
}

int64_t resident_pairs(const void* kernel, int threads, size_t smem) {
  const int64_t most = num_sms() / 2;
  const int dev = current_device();
  std::lock_guard<std::mutex> lk(g_fact_mu);
  KernelFact& f = fact_of(kernel, dev);
  if (!f.pairs) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(2 * most));
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess || clusters <= 0) {
      cudaGetLastError();
      return most;
    }
    f.pairs = std::min<int64_t>(most, clusters);
  }
  return f.pairs;
}

// mode: 0 residues (tensor cores), 1 magnitude (tensor cores),
//       2 residues (SIMT reference), 3 magnitude (SIMT reference).
cudaError_t launch_plane_gemm(int64_t m, int64_t n, int64_t k_pad, const Oz2Moduli& mods,
                              const uint8_t* planes_a, const uint8_t* planes_b, int mode,
                              int16_t* residues, int64_t ldr, float* urow, int* u_max, Oz2Device* dev,
                              cudaStream_t st, int16_t* partials, size_t partial_bytes, const MagnitudeSplit* split, bool fastest) {
  if (m == 0 || n == 0) return cudaSuccess;
  EpiCtx ctx{residues, urow, u_max, dev, m, n, ldr, nullptr, 0};
  if (mode >= 2) {
    dim3 g(static_cast<unsigned>((m + 127) / 128), static_cast<unsigned>(n));
    count_launch();
    if (mode == 2) plane_gemm_simt_kernel<0><<<g, 128, 0, st>>>(planes_a, planes_b, mods, k_pad, ctx);
    else plane_gemm_simt_kernel<1><<<g, 128, 0, st>>>(planes_a, planes_b, mods, k_pad, ctx);
    return cudaGetLastError();
  }
  CUtensorMap ta, tb;
  const bool maps = mode == 0 ? make_block_map(&ta, planes_a, m, k_pad, mods.nplanes) &&
                                    make_block_map(&tb, planes_b, n, k_pad, mods.nplanes)
                              : make_plane_map(&ta, planes_a, m, k_pad) && make_plane_map(&tb, planes_b, n, k_pad);
  if (!maps) return cudaErrorInvalidValue;
  UnitMap um;
  um.ntm = (m + kTileM - 1) / kTileM;
  um.ntn = (n + kTileN - 1) / kTileN;
  um.ntiles = um.ntm * um.ntn;
  um.nunits = um.ntiles * (mode == 0 ? mods.r : 1);
  // Square moduli lead the set; the nonsquare ones are scheduled first.
  um.nsq = 0;
  while (um.nsq < mods.r && mods.sq_base[um.nsq]) ++um.nsq;
  um.nheavy = mode == 0 ? mods.r - um.nsq : 0;
  for (int i = um.nsq; i < mods.r; ++i)
    if (mods.sq_base[i]) um.nheavy = 0;  // not a prefix: keep the index order
  um.ksteps = k_pad / kBK;
  um.kparts = 1;
  um.kpart_steps = um.ksteps;
  const size_t smem = gemm_smem_bytes();
  auto kern = mode == 1 ? plane_gemm_kernel<1> : k_pad == kBK ? plane_gemm_kernel<0> : residue_gemm_kernel<kTileN>;
  cudaError_t err = allow_smem(reinterpret_cast<const void*>(kern), smem);
  if (err != cudaSuccess) return err;
  // Persistent grid: as many CTA pairs as can be resident at once.
  int64_t pairs = resident_pairs(reinterpret_cast<const void*>(kern), kGemmThreads, smem);
  // Split K where the scratch holds the parts (16-byte aligned rows: the
  // fold reads and writes 8 residues at a time).
  if (mode == 0 && partials && reinterpret_cast<uintptr_t>(partials) % 16 == 0 &&
      reinterpret_cast<uintptr_t>(residues) % 16 == 0) {
    const int nheavy_sq = um.nheavy ? um.nsq : mods.r;  // the model's squares
    um.kparts = residue_gemm_kparts(m, n, k_pad, mods.r, nheavy_sq, ldr, partial_bytes, pairs);
    if (fastest && ldr % 8 == 0) {
      const size_t part_bytes = static_cast<size_t>(mods.r) * n * ldr * sizeof(int16_t);
      um.kparts = fastest_kparts(um.ntiles, mods.r, um.ksteps, pairs, m, n,
                                 std::min<int64_t>(kMaxKParts, static_cast<int64_t>(partial_bytes / part_bytes)));
    }
    um.kpart_steps = (um.ksteps + um.kparts - 1) / um.kparts;
    um.nunits *= um.kparts;
    if (um.kparts > 1) ctx.res = partials;
  }
  // The magnitude GEMM of a small C with a long k: parts of k, with U's
  // partial sums (zeroed by the caller) in `split`.
  if (mode == 1 && split && split->parts > 1) {
    um.kparts = split->parts;
    um.kpart_steps = (um.ksteps + um.kparts - 1) / um.kparts;
    um.nunits *= um.kparts;
    kern = plane_gemm_kernel<1, true>;  // same shared memory and threads, so the same pairs fit
    err = allow_smem(reinterpret_cast<const void*>(kern), smem);
    if (err != cudaSuccess) return err;
    ctx.upart = split->sums;
    ctx.ldu = magnitude_ldu(n);
  }
  // A small C in one part: tiles of 64 columns while their units are one wave
  // (256³: the GEMM stage 15.7 µs in 12 units of 256 columns, 11.8 in 48 of 64).
  const int64_t ntn64 = (n + 63) / 64;
  if (mode == 0 && k_pad > kBK && um.kparts == 1 && um.ntm * ntn64 * mods.r <= pairs) {
    um.ntn = ntn64;
    um.ntiles = um.ntm * um.ntn;
    um.nunits = um.ntiles * mods.r;
    kern = residue_gemm_kernel<64>;  // less shared memory, the same threads: as many pairs fit
    err = allow_smem(reinterpret_cast<const void*>(kern), smem);
    if (err != cudaSuccess) return err;
    if (!make_block_map(&tb, planes_b, n, k_pad, mods.nplanes, 32)) return cudaErrorInvalidValue;
  }
  pairs = std::max<int64_t>(1, std::min<int64_t>(pairs, um.nunits));
  count_launch();
  // The GEMM kernels let no dependent start early: the deconstruction's two
  // blocks per SM, resident beside the "+1" GEMM on the SMs it leaves room on,
  // spread unevenly (16384×16×16384 4172 µs a call, 4408 with the early start;
  // 1024²×65536 2795 and 2873).
  err = launch_dependent(kern, dim3(static_cast<unsigned>(2 * pairs)), dim3(kGemmThreads), smem, st, ta, tb, mods, k_pad,
                         um, ctx);
  if (err == cudaSuccess && ctx.upart) err = launch_plus_one_rowmax(ctx.upart, m, n, ctx.ldu, urow, u_max, st);
  if (err == cudaSuccess && mode == 0 && um.kparts > 1) {  // the residue GEMM's parts, folded into C^(i)
    const int64_t row_threads = (m + 7) / 8;
    dim3 g(static_cast<unsigned>((row_threads + kFoldThreads - 1) / kFoldThreads),
           static_cast<unsigned>(std::min<int64_t>(n, 32768)), static_cast<unsigned>(mods.r));
    count_launch();
    err = launch_dependent(fold_parts_kernel, g, dim3(kFoldThreads), 0, st, partials, residues, m, n, ldr, um.kparts,
                           mods);
  }
  return err;
}

// The rate probe on as many CTA pairs as can be resident at once.
cudaError_t launch_mma_rate(int64_t iters, Oz2Device* dev, int* pairs_out, cudaStream_t st) {
  const void* kern = reinterpret_cast<const void*>(mma_rate_kernel);
  const cudaError_t err = allow_smem(kern, kProbeSmem);
  if (err != cudaSuccess) return err;
  const int64_t pairs = resident_pairs(kern, kProbeThreads, kProbeSmem);
  if (pairs_out) *pairs_out = static_cast<int>(pairs);
  count_launch();
  mma_rate_kernel<<<static_cast<unsigned>(2 * pairs), kProbeThreads, kProbeSmem, st>>>(iters, dev);
  return cudaGetLastError();
}

}  // namespace oz2
