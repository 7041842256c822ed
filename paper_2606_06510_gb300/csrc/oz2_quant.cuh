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

// Ã of an entry as a 64-bit two's complement word, any scale and quantiser.
__device__ __forceinline__ unsigned long long quantise_entry(double x, int d, bool rn) {
  if (!rn && d <= kTzFastMaxD) return quantise_tz(x, d);
  const Split sp = split_double(x);
  const unsigned long long a = quantise_abs(sp, d, rn);
  return sp.neg ? 0ull - a : a;
}

}  // namespace oz2
