// The one rounding of the split path: RN(X 2^k) of an exact integer X to
// binary64 (recombination kernel and the product kernel that recombines).
#pragma once

#include <cstdint>

namespace hs {

// RN(X 2^k) for a 128-bit integer X, ties to even, subnormals and overflow
// handled: the value is rounded once, at the precision its exponent allows.
static __device__ __noinline__ double round_scaled_i128(__int128 X, int k) {
  if (X == 0) return 0.0;
  const bool neg = X < 0;
  unsigned __int128 m = neg ? (unsigned __int128)(-X) : (unsigned __int128)X;
  const unsigned long long hi = (unsigned long long)(m >> 64), lo = (unsigned long long)m;
  const int nb = hi ? 128 - __clzll((long long)hi) : 64 - __clzll((long long)lo);
  const int e = nb - 1 + k;               // exponent of the leading bit
  int ulp = e - 52;                       // exponent of the last kept bit
  if (ulp < -1074) ulp = -1074;
  const int drop = ulp - k;               // low bits of m below the last kept bit
  unsigned long long q;
  if (drop <= 0) {
    q = (unsigned long long)(m << (-drop));   // < 2^53
  } else if (drop > nb) {
    q = 0;                                  // below half of the smallest step
  } else {
    const unsigned __int128 qq = m >> drop;
    const unsigned __int128 rem = m - (qq << drop);
    const unsigned __int128 half = (unsigned __int128)1 << (drop - 1);
    q = (unsigned long long)qq;
    if (rem > half || (rem == half && (q & 1ull))) q += 1;
  }
  if (q == (1ull << 53)) {                 // rounding carried into a new binade
    q >>= 1;
    ulp += 1;
  }
  unsigned long long bits;
  if (q < (1ull << 52)) {
    bits = q;                               // subnormal (ulp == -1074) or zero
  } else {
    const long long biased = (long long)ulp + 1075;
    if (biased >= 2047)
      bits = 0x7FF0000000000000ull;         // overflow rounds to infinity
    else
      bits = ((unsigned long long)biased << 52) | (q & 0xFFFFFFFFFFFFFull);
  }
  if (neg) bits |= 0x8000000000000000ull;
  return __longlong_as_double((long long)bits);
}

// The same for a 64-bit X: 64-bit integer work when the result is normal (the
// common case); anything else goes to the general routine.
__device__ __forceinline__ double round_scaled64(long long X, int k) {
  if (X != 0) {
    const bool neg = X < 0;
    const unsigned long long m = neg ? 0ull - (unsigned long long)X : (unsigned long long)X;
    const int nb = 64 - __clzll((long long)m);
    const int drop = nb - 53;
    unsigned long long q;
    int ulp;
    if (drop <= 0) {
      q = m << (-drop);
      ulp = k + drop;
    } else {
      q = (m + ((1ull << (drop - 1)) - 1ull) + ((m >> drop) & 1ull)) >> drop;
      ulp = k + drop;
      if (q == (1ull << 53)) {
        q >>= 1;
        ulp += 1;
      }
    }
    const int biased = ulp + 1075;
    if (biased >= 1 && biased <= 2046) {
      const unsigned long long bits = ((unsigned long long)biased << 52) |
                                      (q & 0xFFFFFFFFFFFFFull) |
                                      (neg ? 0x8000000000000000ull : 0ull);
      return __longlong_as_double((long long)bits);
    }
  }
  return round_scaled_i128((__int128)X, k);
}

__device__ __forceinline__ double round_scaled(__int128 X, int k) {
  const long long lo = (long long)X;
  if ((__int128)lo == X) return round_scaled64(lo, k);
  return round_scaled_i128(X, k);
}

// The forms below give the same value as round_scaled64 where
// kScaleLo <= k <= kScaleHi (every |X| >= 1 then gives a normal result), for the
// product kernel's epilogue, which rounds 16384 entries a tile.  One leaves the
// rounding to the conversion instruction (8192 cycles a tile on the binary64
// unit, few instructions), the other is about 20 integer instructions
// (round_scaled64: 9900 cycles a tile); used in turn they keep both units busy.
constexpr int kScaleLo = -1022, kScaleHi = 960;
__device__ __forceinline__ double round_scaled_cvt(long long X, int k) {
  const double d = (double)X;
  const int hi = __double2hiint(d);
  return __hiloint2double(hi == 0 ? 0 : hi + (int)((unsigned)k << 20), __double2loint(d));
}

__device__ __forceinline__ double round_scaled_int(long long X, int k) {
  const int sgn = (int)(X >> 63);
  const unsigned long long m = (unsigned long long)((X ^ (X >> 63)) - (X >> 63));
  const uint32_t mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
  if (mh == 0) return round_scaled_cvt(X, k);
  const int n = __clz((int)mh);
  const uint32_t h = __funnelshift_l(ml, mh, n), l = ml << n;   // leading bit at 63
  uint32_t qh = h >> 11, ql = __funnelshift_r(l, h, 11);
  // half to even: up when the 11 dropped bits and the last kept one exceed half
  const uint32_t up = ((l & 0x7FFu) + (ql & 1u) + 0x3FFu) >> 11;
  ql += up;
  qh += (ql < up ? 1u : 0u) + ((uint32_t)(1085 - n + k) << 20);   // the leading bit adds one
  return __hiloint2double((int)(qh | ((uint32_t)sgn & 0x80000000u)), (int)ql);
}

// RN((X 2^HS + low) 2^k) for 0 <= low < 2^HS and k from kScaleLo to kScaleHi - 32,
// in 32-bit words: the sum's 64 leading bits, the ones below folded into the last
// of them (round to odd), are left to the conversion to round.  The integer
// units run at half the issue rate, so that this form, 20 instructions and 64
// cycles a warp on the binary64 unit, is bound by the latter; all in integers it
// took 41 instructions.
template <int HS>
__device__ __forceinline__ double round_scaled_ext(unsigned long long X, uint32_t low, int k) {
  static_assert(HS > 0 && HS < 31, "three words, shifts below 32");
  const uint32_t xl = (uint32_t)X, xh = (uint32_t)(X >> 32);
  const uint32_t s0 = xl * (1u << HS) + low, s1 = __funnelshift_l(xl, xh, HS);
  const int s2 = (int)xh >> (32 - HS);
  const uint32_t sgn = (uint32_t)(s2 >> 31);
  // the bits that 64 cannot hold: of the words above the sign copies
  const int z = __clz((int)__funnelshift_l(s1 ^ sgn, (uint32_t)s2 ^ sgn, 1)), n = 32 - z;
  const uint32_t lost = __funnelshift_lc(0u, s0, z);
  const uint32_t t0 = __funnelshift_r(s0, s1, n) | (lost ? 1u : 0u);
  const uint32_t t1 = __funnelshift_r(s1, (uint32_t)s2, n);
  return round_scaled_cvt((long long)(((unsigned long long)t1 << 32) | t0), k + n);
}

}  // namespace hs
