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

}  // namespace hs
