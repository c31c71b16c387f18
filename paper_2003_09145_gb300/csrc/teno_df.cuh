// teno_df.cuh -- numbers held as the sum of two binary32 values (h + l), for
// host and device: about 46 bits of precision at FP32 rates.
//
// GB300 issues one FP64 warp instruction per 64 cycles and SM partition,
// whatever its lanes do, and an FP32 one every 2.  The closed-form flux needs
// its Roe state only inside the correction terms, which are multiplied by U~
// (a sixtieth of the fifth difference of the state): where these terms stay
// below 2^-7 of the flux scale, an error of 2^-43 of them is below 2^-50 of
// the flux scale at worst, and far below it in smooth flow -- no more than
// the rounding of a binary64 chain of the flux itself.  So these terms run in
// two binary32 values (closed_df_rough tests each interface) and the 53-bit
// arithmetic is left to the sums that need it.
//
// The operations keep h and l unnormalised between them (|l| up to a few
// ulps of h after a product, more after a cancelling sum): every product
// carries both cross terms, so only l_a l_b (2^-46 relative to the operands'
// scales) and the roundings of the low parts (2^-24 of a low part each) are
// lost.  Every FP32 operation is written with its rounding explicit.
#pragma once

#include "teno_cert.cuh"
#include "teno_fixsum.cuh"

namespace teno_df {

using teno_cert::fadd;
using teno_cert::ffma;
using teno_cert::fmul;
using teno_cert::fsub;

struct df {
  float h, l;
};

TENO_CERT_HD uint32_t bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, sizeof(b));
  return b;
#endif
}
TENO_CERT_HD float from_bits(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, sizeof(x));
  return x;
#endif
}

// 2^k as binary32 from its biased exponent field, 0 below the normal range
TENO_CERT_HD float pow2_field(int f) { return from_bits(static_cast<uint32_t>(f < 0 ? 0 : f) << 23); }

TENO_CERT_HD df neg(df a) { return {-a.h, -a.l}; }
// exact scaling by a power of two
TENO_CERT_HD df scale(df a, float p) { return {fmul(a.h, p), fmul(a.l, p)}; }

// x truncated to 46 bits (24 in h, the next 23 in l), 2^-100 <= |x| < 2^127
TENO_CERT_HD df split(double x) {
  const uint32_t hi = teno_fix::hi_word(x), lo = teno_fix::lo_word(x);
  const uint32_t m = hi << 1;
  const uint32_t h = (m * 4u - (896u << 23)) | (hi & 0x80000000u) | (lo >> 29);
  const uint32_t b = (h & 0xFF800000u) - (23u << 23);   // the low part's unit, with the sign
  const uint32_t r = (lo >> 6) & 0x7FFFFFu;
  return {from_bits(h), fsub(from_bits(b | r), from_bits(b))};
}
// the same; magnitudes below 2^-100 become 0 (a direction at rest stays at
// rest exactly)
TENO_CERT_HD df from_double(double x) {
  const df d = split(x);
  const bool zero = (teno_fix::hi_word(x) & 0x7FFFFFFFu) < (923u << 20);
  return {zero ? 0.0f : d.h, zero ? 0.0f : d.l};
}

TENO_CERT_HD df add(df a, df b) {
  const float s = fadd(a.h, b.h), t = fsub(s, a.h);
  const float e = fadd(fsub(a.h, fsub(s, t)), fsub(b.h, t));
  return {s, fadd(e, fadd(a.l, b.l))};
}

TENO_CERT_HD df mul(df a, df b) {
  const float p = fmul(a.h, b.h);
  return {p, ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)))};
}

TENO_CERT_HD df sqr(df a) {
  const float p = fmul(a.h, a.h);
  return {p, ffma(2.0f * a.h, a.l, ffma(a.h, a.h, -p))};
}

// (the host's seeds are rounded to nearest; a test may move them by what the
// instructions may be off: one ulp, and 2^-22.9)
#ifndef TENO_HOST_SEED
#define TENO_HOST_SEED(y, ulps) (y)
#endif
TENO_CERT_HD float rcp_seed(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return TENO_HOST_SEED(1.0f / x, 1);
#endif
}
TENO_CERT_HD float rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return TENO_HOST_SEED(1.0f / std::sqrt(x), 2);
#endif
}

// 1/a: one third-order step y (1 + e + e^2), e = 1 - a y, from a seed within
// a few ulps (|e| < 2^-21, so e^3 is lost)
TENO_CERT_HD df recip(df a) {
  const float y = rcp_seed(a.h);
  const float e = ffma(-a.l, y, ffma(-a.h, y, 1.0f));
  return {y, fmul(y, ffma(e, e, e))};
}

// 1/sqrt(a): y (1 + e/2 + 3 e^2/8), e = 1 - a y^2
TENO_CERT_HD df rsqrt(df a) {
  const float y = rsqrt_seed(a.h);
  const float z = fmul(y, y), ze = ffma(y, y, -z);
  const float e = ffma(-a.l, z, ffma(-a.h, ze, ffma(-a.h, z, 1.0f)));
  return {y, fmul(y, fmul(e, ffma(0.375f, e, 0.5f)))};
}

// A 2^(E - 1078), the value of a fixed-point sum (teno_fixsum.cuh), to 48
// bits; values below 2^-92 of a component with E <= 930 become 0
TENO_CERT_HD df from_fixed(int64_t A, uint32_t E) {
  const float c2 = static_cast<float>(static_cast<int32_t>(A >> 42));
  const float c1 = static_cast<float>(static_cast<int32_t>((A >> 21) & 0x1FFFFF));
  const float c0 = static_cast<float>(static_cast<int32_t>(A & 0x1FFFFF));
  const float s = fmul(c2, 0x1p21f);
  const float h = fadd(s, c1);                       // unit 2^21
  const float l = ffma(fsub(c1, fsub(h, s)), 0x1p21f, c0);
  const int f = static_cast<int>(E) - 951;           // 2^(E - 1078) has the field E - 951
  return {fmul(h, pow2_field(f + 21)), fmul(l, pow2_field(f))};
}

// h + l in binary64 with integer operations, to 2^-46 relative (and 2^-125, as
// l ends at 2^-126 and smaller values become 0): h + l is renormalised, h
// moved one ulp towards zero where l points back (l then rounds once), and l's
// significand, shifted to h's exponent, fills the result's low 29 bits.  (Two FP64 additions of the widened parts would hold the FP64
// pipe for 128 cycles a warp; this is some 20 instructions.)
TENO_CERT_HD double to_double(df a) {
  const float s = fadd(a.h, a.l), t = fsub(s, a.h);
  float l = fadd(fsub(a.h, fsub(s, t)), fsub(a.l, t));
  uint32_t hb = bits(s);
  if ((hb & 0x7FFFFFFFu) < (2u << 23)) return 0.0;
  const bool back = l != 0.0f && ((bits(l) ^ hb) >> 31);
  const float h = from_bits(hb - (back ? 1u : 0u));
  l = fadd(l, fsub(s, h));
  hb = bits(h);
  const uint32_t mag = hb & 0x7FFFFFFFu;
  // |l| / 2^(e - 52) with e the exponent of h: its 24-bit significand times
  // 2^(e_l - e + 29), e_l <= e - 23
  const uint32_t lm = bits(l) & 0x7FFFFFFFu, el = lm >> 23;
  const uint32_t sh = (mag >> 23) - el - 23u;
  uint32_t q = ((lm & 0x7FFFFFu) | 0x800000u) << 6 >> (sh < 31u ? sh : 31u);
  q = el == 0u ? 0u : (q > 0x1FFFFFFFu ? 0x1FFFFFFFu : q);
  const uint32_t hi = (hb & 0x80000000u) | ((mag >> 3) + (896u << 20));
  const uint32_t lo = (mag << 29) | q;
  return teno_fix::from_bits((static_cast<uint64_t>(hi) << 32) | lo);
}

}  // namespace teno_df
