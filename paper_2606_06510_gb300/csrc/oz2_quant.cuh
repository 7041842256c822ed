// Quantisation of one entry (Eq. scale; Algorithm 1 "lin:quant"), shared by
// the deconstruction and the kernels that multiply the integers' digits.
#pragma once

#include "oz2_common.cuh"

namespace oz2 {

// Integer significand M and exponent x with |x| = M·2^x (M < 2^53), or M = 0.
struct Split {
  unsigned long long M;
  int ex;
  bool neg;
};
__device__ __forceinline__ Split split_double(double v) {
  unsigned long long b = __double_as_longlong(v);
  Split s;
  s.neg = (b >> 63) != 0;
  int E = static_cast<int>((b >> 52) & 0x7FF);
  unsigned long long mant = b & ((1ull << 52) - 1);
  if (E == 0x7FF) {  // non-finite entries only occur in rows zeroed by the flags
    s.M = 0;
    s.ex = 0;
  } else if (E == 0) {
    s.M = mant;
    s.ex = -1074;
  } else {
    s.M = mant | (1ull << 52);
    s.ex = E - 1075;
  }
  return s;
}

// ⌊2^d |v|⌉ (TZ: toward zero, RN: half to even) as an unsigned integer; the
// scale choice guarantees the result is below 2^62.
__device__ __forceinline__ unsigned long long quantise_abs(const Split& s, int d, bool rn) {
  if (s.M == 0) return 0;
  int sh = s.ex + d;
  if (sh >= 0) return s.M << min(sh, 63);
  int r = -sh;
  if (r >= 64) return 0;  // < 2^53·2^-64 < 1/2
  unsigned long long q = s.M >> r;
  if (rn) {
    unsigned long long rem = s.M & ((1ull << r) - 1);
    unsigned long long half = 1ull << (r - 1);
    if (rem > half || (rem == half && (q & 1))) ++q;
  }
  return q;
}

// Truncating quantisation (Eq. scale, TZ): Ã = trunc(x·2^d) as a 64-bit two's
// complement word, for rows with d ≤ kTzFastMaxD.  With x = ±M·2^(sh - d),
// M < 2^53, Ã = ±⌊M·2^10 / 2^(10 - sh)⌋: the significand is shifted up by 10
// (below 2^63) and then right by r = 10 - sh with one clamping 64-bit shift, so
// zeros, subnormals and entries that shift out entirely need no branch.  That needs sh ≤ 9: a normal x has M ≥ 2^52
// and |Ã| < 2^62, and a subnormal one has sh = d - 1074 ≤ 9 for
// d ≤ kTzFastMaxD (rows with a larger scale, whose largest entry is itself
// subnormal, take the general path).  d = -4096 gives Ã = 0 for any x.
constexpr int kTzFastMaxD = 1083;
__device__ __forceinline__ unsigned long long quantise_tz(double x, int d) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const uint32_t E = (hi >> 20) & 0x7FFu;
  const uint32_t mh = (min(E, 1u) << 20) + (hi & 0xFFFFFu);  // M = mh·2^32 + lo
  const uint32_t r = static_cast<uint32_t>(10 + 1075 - d) - max(E, 1u);
  const unsigned long long m10 = (static_cast<unsigned long long>(__funnelshift_l(lo, mh, 10)) << 32) | (lo << 10);
  unsigned long long q;
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(m10), "r"(r));
  const uint32_t sgn = static_cast<uint32_t>(static_cast<int>(hi) >> 31);  // 0 or all ones
  return ((static_cast<unsigned long long>(static_cast<uint32_t>(q >> 32) ^ sgn) << 32) |
          (static_cast<uint32_t>(q) ^ sgn)) + (sgn & 1u);
}

// ⌈log2 |v|⌉ for finite nonzero v.
__device__ __forceinline__ int ceil_log2_abs(const Split& s) {
  int bl = 64 - __clzll(static_cast<long long>(s.M));
  bool pow2 = (s.M & (s.M - 1)) == 0;
  return s.ex + (pow2 ? bl - 1 : bl);
}

// E4M3 code of 2^q, q ∈ [-9, 0] (subnormal below 2^-6).
__device__ __forceinline__ uint32_t e4m3_pow2(int q) {
  return q >= -6 ? static_cast<uint32_t>((q + 7) << 3) : (1u << (q + 9));
}

// Magnitude-plane code of x: 0 for x = 0, else the E4M3 code of
// 2^max(-c, ⌈log2|x|⌉ - ex).  A normal double has ⌈log2|x|⌉ = E - 1023, plus
// one when its fraction is nonzero, read off the high word; subnormals take
// the general path.
__device__ __forceinline__ uint32_t magnitude_code(double x, int ex, int c) {
  const unsigned long long b = __double_as_longlong(x);
  const uint32_t hi = static_cast<uint32_t>(b >> 32), lo = static_cast<uint32_t>(b);
  const int E = static_cast<int>((hi >> 20) & 0x7FFu);
  const bool frac = ((hi & 0xFFFFFu) | lo) != 0;
  if (E == 0x7FF) return 0u;  // non-finite entries only occur in rows zeroed by the flags
  if (E == 0) {
    if (!frac) return 0u;
    const Split sp = split_double(x);
    return e4m3_pow2(max(-c, ceil_log2_abs(sp) - ex));
  }
  return e4m3_pow2(max(-c, E - 1023 + (frac ? 1 : 0) - ex));
}

// The clamp c of the magnitude planes for this k (reading R-scale): the sums of
// the "+1" GEMM are integers in units of 2^-2c and stay below 2^24.
inline int magnitude_clamp(int64_t k) {
  const int lk = k <= 1 ? 0 : 64 - __builtin_clzll(static_cast<unsigned long long>(k - 1));
  const int c = (24 - lk) / 2;
  return c < 0 ? 0 : (c > kMagClampMax ? kMagClampMax : c);
}

// Ã of an entry as a 64-bit two's complement word, any scale and quantiser.
__device__ __forceinline__ unsigned long long quantise_entry(double x, int d, bool rn) {
  if (!rn && d <= kTzFastMaxD) return quantise_tz(x, d);
  const Split sp = split_double(x);
  const unsigned long long a = quantise_abs(sp, d, rn);
  return sp.neg ? 0ull - a : a;
}

}  // namespace oz2
