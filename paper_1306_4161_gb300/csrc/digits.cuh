// The S digits of a value of the split path (slicing kernels).
//
// With F = floor(|x| 2^-e 2^64) (below 2^63, since the exponent scan makes
// |x| 2^-e < 1/2; a bit dropped below F is or-ed into bit 0 of F, which is never a
// digit or rounding bit) and Y_s = RN(F / 2^(p+1)), p = 63 - W s (ties to even),
// digit s is t_s = Y_s - 2^W Y_(s-1): the closed form of the Ozaki splitting
// r <- r 2^W - rint(r 2^W) (shifting by the even integer 2^W t does not change a
// half-to-even decision).  A negative x has the negated digits.
//
// The digits come out of fp32 arithmetic, whose units are free here and run at
// twice the rate of the integer ones (in integers a value of 5 digits took 68
// instructions on the integer pipe, which bound the kernels).  The remainder after
// digit s is at most 2^p, so with 23 more bits of F and one bit that says whether
// any below is set (round to odd: below every rounding bit that is still to come
// from this window) it is exact in fp32, and the next digits are its roundings: an
// add of 1.5 2^23 rounds to an integer, ties to even.  When the next rounding bit
// would lie below the window, the bits that follow are added and the "any" bit
// taken out again.
#pragma once

#include <cstdint>

namespace hs {

struct Fixed64 {
  uint32_t h, l;   // F
};

// eb = e + 1011: then |x| 2^-e 2^64 = m 2^sh with sh = max(E, 1) - eb, for the
// significand m (hidden bit included) and the biased exponent E of x.  Beside the
// common case, 0 <= sh < 32: values more than 2^11 below the row's largest,
// subnormals and zeros; also whatever a non-finite input gives, which the exponent
// scan has reported.
static __device__ __noinline__ uint2 fixed_rare(uint32_t hi, uint32_t lo, int eb) {
  const int E = (int)((hi >> 20) & 0x7FFu), sh = max(E, 1) - eb;
  const uint32_t mhi = (hi & 0xFFFFFu) | (E ? 0x100000u : 0u);
  uint32_t h, l, dropped = 0u;
  if (sh >= 32) {
    h = __funnelshift_lc(0u, lo, (unsigned)(sh - 32));    // lo << (sh - 32), 0 past 63
    l = 0u;
  } else if (sh >= 0) {
    h = __funnelshift_l(lo, mhi, (unsigned)sh);
    l = lo << sh;
  } else if (sh > -32) {
    const unsigned r = (unsigned)(-sh);                   // 1..31
    h = mhi >> r;
    l = __funnelshift_r(lo, mhi, r);
    dropped = lo << (32u - r);
  } else if (sh > -64) {
    const unsigned r = (unsigned)(-sh) - 32u;             // 0..31
    h = 0u;
    l = mhi >> r;
    dropped = lo | __funnelshift_lc(0u, mhi, 32u - r);    // the low r bits of mhi
  } else {
    h = l = 0u;
    dropped = mhi | lo;
  }
  return make_uint2(h, l | (dropped != 0u ? 1u : 0u));
}

__device__ __forceinline__ Fixed64 fixed64(double x, int eb) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int sh = (int)((hi >> 20) & 0x7FFu) - eb;
  // (with eb > 0 a biased exponent of 0 has sh < 0)
  if ((unsigned)sh < (eb > 0 ? 32u : 0u))
    return {__funnelshift_l(lo, (hi & 0xFFFFFu) | 0x100000u, (unsigned)sh), lo << sh};
  const uint2 F = fixed_rare(hi, lo, eb);
  return {F.x, F.y};
}

constexpr float kRoundMagic = 12582912.0f;        // 1.5 2^23
__host__ __device__ constexpr float exp2i(int n) {
  float v = 1.0f;
  for (; n > 0; --n) v *= 2.0f;
  for (; n < 0; ++n) v *= 0.5f;
  return v;
}

// Digits s..S from r 2^mul, their remainder in units of digit s's last place (the
// window's bits end at `slot`, whose place `any` holds).
template <int W, int S, int s, int slot, int mul>
__device__ __forceinline__ void digits_from(float r, uint32_t any, const Fixed64 &F, float sgn,
                                            float (&t)[S]) {
  constexpr int p = 63 - W * s;
  constexpr float c = exp2i(mul);
  t[s - 1] = __fadd_rn(__fmaf_rn(r, c, kRoundMagic), -kRoundMagic);
  if constexpr (s < S) {
    r = __fmaf_rn(r, c, -t[s - 1]);
    if constexpr (p - W > slot) {
      digits_from<W, S, s + 1, slot, W>(r, any, F, sgn, t);
    } else {
      // the next window: bits [ns + 1, slot], and whether any of [0, ns] is set
      constexpr int ns = p > 23 ? p - 23 : 0;
      static_assert(ns < 31 && slot - ns < 22 && p - W > ns, "23 bits more");
      constexpr uint32_t field = (1u << (slot - ns + 1)) - 1u;
      const uint32_t v = ns ? __funnelshift_r(F.l, F.h, ns) : F.l;
      const uint32_t below = ns && (F.l & ((2u << ns) - 1u)) ? 1u : 0u;
      const int w = (int)((v & (ns ? field & ~1u : field)) | below) - (int)(any << (slot - ns));
      const float f = __fadd_rn(__int_as_float(0x4B400000 + w), -kRoundMagic);
      r = __fmaf_rn(f, sgn * exp2i(ns - p - 1), r);
      digits_from<W, S, s + 1, ns, W>(r, below, F, sgn, t);
    }
  }
}

template <int W, int S>
__device__ __forceinline__ void digits(double x, int eb, float (&t)[S]) {
  static_assert(W >= 7 && W <= 9 && W * S <= 56, "windows as below; the last rounding bit is 7");
  const Fixed64 F = fixed64(x, eb);
  const float sgn = __int_as_float((__double2hiint(x) & (int)0x80000000) | 0x3F800000);
  constexpr int slot = 40;   // the first window: bits 62..41
  const uint32_t any = (F.h & 0x1FFu) | F.l ? 1u : 0u;
  const uint32_t v = ((F.h >> 8) & ~1u) | any;
  const float f = __fadd_rn(__int_as_float((int)(0x4B000000u | v)), -8388608.0f);
  digits_from<W, S, 1, slot, slot - (64 - W)>(f * sgn, any, F, sgn, t);
}

}  // namespace hs
