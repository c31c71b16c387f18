// teno_closed_core.cuh -- the arithmetic of the closed form that runs in two
// binary32 values (teno_df.cuh), for host and device: the cells' and the
// speeds' binary32 forms, the Roe state, the certificate's view of it, the
// corrections, and the tests that say where these forms hold (elsewhere
// teno_closed.cuh takes binary64).
#pragma once

#include "teno_df.cuh"

namespace teno {

using teno_cert::CertIfc;

// x rounded to binary32 (to nearest, halves away from zero) by integer
// operations, for 2^-126 <= |x| < 2^127; smaller magnitudes become 2^-126 (and up
// to eight ulps), larger ones, infinities and NaN a value just below 2^128, as
// hi_float's.  (Without a branch, which would keep the next value's load from
// starting.)
TENO_CERT_HD float near_float(double x) {
  const uint32_t hi = teno_fix::hi_word(x), lo = teno_fix::lo_word(x);
  uint32_t m = hi & 0x7FFFFFFFu;
  m = m < (897u << 20) ? (897u << 20) : m;
  m = m > ((1150u << 20) | 0xFFFFEu) ? ((1150u << 20) | 0xFFFFEu) : m;
  return teno_df::from_bits((((m - (896u << 20)) << 3) + (((lo >> 28) + 1u) >> 1)) | (hi & 0x80000000u));
}

// The same by two binary32 values (halves to even), for the speeds: with its
// branch the closed-form pass is scheduled better (13.6 against 13.9 ms of a 256^3
// step's fluxes).
TENO_CERT_HD float near_speed(double x) {
  const uint32_t e = (teno_fix::hi_word(x) >> 20) & 0x7FFu;
  if (e - 923u >= 200u) return teno_cert::hi_float(x);
  const teno_df::df d = teno_df::split(x);
  return teno_cert::fadd(d.h, d.l);
}

// The speeds in the forms the closed form reads: halved, as two binary32
// values (the middle one, and the sum and difference of the acoustic
// ones' differences against it -- closed_out's amid, sg, df), as binary32, and
// whether they lie in the range of teno_df's terms (2^-19 .. 2^30).
struct FaceSpeeds {
  teno_df::df amid, sg, dd;
  float ha[3], amax;
  bool in_range;
};
TENO_CERT_HD FaceSpeeds face_speeds(const double (&a3)[3]) {
  using namespace teno_df;
  FaceSpeeds F;
  const df am = from_double(a3[0]), a0 = from_double(a3[1]), ap = from_double(a3[2]);
  const df d0 = add(am, neg(a0)), dE = add(ap, neg(a0));
  F.amid = a0;
  F.sg = add(d0, dE);
  F.dd = add(d0, neg(dE));
#pragma unroll
  for (int s = 0; s < 3; ++s) F.ha[s] = near_speed(a3[s]);
  F.amax = 2.0f * fmaxf(F.ha[0], F.ha[2]);
  F.in_range = F.amax >= 0x1p-19f && F.amax <= 0x1p30f;
  return F;
}

// The Roe state in two binary32 values, from the cells' sqrt(rho),
// (E+p)/sqrt(rho) and m_k/sqrt(rho) (roe_interface's average): u~, |u~|^2, H~,
// c~^2 and 1/c~.
template <int NDIM>
struct RoeDf {
  teno_df::df u[NDIM], q2, H, c2, ic;
  float um;    // the largest average of |u_k| (the scale of u~'s rounding)
  bool sums;   // the averages' sums are far above from_double's floor of 2^-100
};
template <int NDIM>
struct RoeCellDf {   // one cell's contribution
  teno_df::df sr, sh, su[NDIM];
};
template <int NDIM>
TENO_CERT_HD RoeCellDf<NDIM> roe_cell(double sr, double sh, const double (&su)[NDIM]) {
  RoeCellDf<NDIM> R;
  R.sr = teno_df::from_double(sr);
  R.sh = teno_df::from_double(sh);
#pragma unroll
  for (int k = 0; k < NDIM; ++k) R.su[k] = teno_df::from_double(su[k]);
  return R;
}
// (gm1: gamma - 1 as two binary32 values)
template <int NDIM>
TENO_CERT_HD void roe_df(const RoeCellDf<NDIM>& a, const RoeCellDf<NDIM>& b, teno_df::df gm1, RoeDf<NDIM>& R) {
  using namespace teno_df;
  const df sr = add(a.sr, b.sr), sh = add(a.sh, b.sh);
  R.sums = sr.h >= 0x1p-40f && sh.h >= 0x1p-40f;
  const df y = recip(sr);
  R.um = 0.0f;
#pragma unroll
  for (int k = 0; k < NDIM; ++k) {
    R.u[k] = mul(add(a.su[k], b.su[k]), y);
    R.q2 = k == 0 ? sqr(R.u[0]) : add(R.q2, sqr(R.u[k]));
    R.um = fmaxf(R.um, fadd(fabsf(a.su[k].h), fabsf(b.su[k].h)));
  }
  R.um = fmul(R.um, y.h);
  R.H = mul(sh, y);
  R.c2 = mul(gm1, add(R.H, scale(R.q2, -0.5f)));
  R.ic = teno_df::rsqrt(R.c2);
}
// Where the Roe state is good to 2^-44 of its terms: c~^2 keeps 2^-6 of
// (gamma - 1) H~ (Mach numbers below about 18 for gamma = 1.4; c~^2 is then
// good to 2^-38), and the sums lie above 2^-40, so that the absolute 2^-100 of
// from_double stays below 2^-58 of sqrt(rho) and H~ and, as c~^2 >= 2^-6 (gamma
// - 1) H~, below 2^-55 (gamma - 1)^(-1/2) of c~ in u~.
template <int NDIM>
TENO_CERT_HD bool roe_df_ok(const RoeDf<NDIM>& R, teno_df::df gm1) {
  return R.sums && R.c2.h > 0x1p-6f * gm1.h * R.H.h;
}

// The certificate's view of that Roe state, rounded to binary32, where
// roe_df_ok holds.
template <int NDIM, int DIR>
TENO_CERT_HD void cert_begin_df(const RoeDf<NDIM>& R, const float (&ha3)[3], teno_df::df gm1, CertIfc<NDIM>& C) {
  using teno_cert::fadd;
  using teno_cert::fmul;
  float uf[NDIM], ha[NDIM + 2];
#pragma unroll
  for (int k = 0; k < NDIM; ++k) uf[k] = fadd(R.u[k].h, R.u[k].l);
#pragma unroll
  for (int f = 0; f < NDIM + 2; ++f) ha[f] = ha3[f == 0 ? 0 : (f == NDIM + 1 ? 2 : 1)];
  const float ic = fadd(R.ic.h, R.ic.l);
  const float hb1 = fmul(0.5f * gm1.h, fmul(ic, ic));
  teno_cert::cert_begin_f<NDIM, DIR>(uf, hb1, fmul(0.5f * hb1, fadd(R.q2.h, R.q2.l)), 0.5f * ic, ha,
                                     teno_cert::kCertRounded, C);
}

// The stencil's largest density and energy between 2^-20 and 2^30, and 2^-40
// and 2^95: every term of the test and of teno_df then lies in binary32's range
// (|u| and c are bounded by the speeds), and the floors of the conversions
// (2^-86 in U~, 2^-125 in a correction) far below the flux scale.
TENO_CERT_HD bool df_range(float rho_max, float e_max) {
  return rho_max >= 0x1p-20f && rho_max < 0x1p30f && e_max >= 0x1p-40f && e_max < 0x1p95f;
}

// Whether the corrections in two binary32 values could be off by more than
// 2^-50 of the flux scale (alpha rho, alpha^2 rho, alpha E: alpha the largest
// speed, rho and E the stencil's largest), a bound like that of the binary64
// chains that they are added to (five roundings of terms up to 3 F each).  With
// eps = 2^-43 the error against the terms' magnitudes (a few operations of
// 2^-45, and 1/c~ of 2^-44), u~ is off by eps um (um: the cells' average |u_k|,
// which u~ may cancel against), c~^2 and 1/c~ by eps g with g = (gamma - 1) H~ /
// c~^2 (um^2 <= 2 H~, so that u~'s share is in it), closed_df's T and V by eps A
// and eps B below, t + V by eps g W, c~ ngd by eps g alpha W and gs by eps g
// alpha G; the sums U~ add their floor of 2^-86 = eps 2^-43.  (The factors 1/c~
// count: in a cold region alpha / c~ is large where the speeds are set
// elsewhere.)  Ut: 60 U~.  Against a test of U~ alone it costs a 256^3 step 21.06 ->
// 21.29 ms, a 2048^2 one 3.38 -> 3.44 ms.
constexpr float kRoughLimit = 30.0f * 0x1p-7f;
template <int NDIM, int DIR>
TENO_CERT_HD bool closed_df_rough(const teno_df::df (&Ut)[NDIM + 2], const RoeDf<NDIM>& R, teno_df::df gm1, float amax,
                                  float rho_max, float e_max) {
  using namespace teno_df;
  constexpr int NVAR = NDIM + 2;
  constexpr float floor_u = 0x1p-43f;
  const float a0 = fadd(fabsf(Ut[0].h), floor_u), aE = fadd(fabsf(Ut[NVAR - 1].h), floor_u);
  float as = 0.0f, am = 0.0f;
#pragma unroll
  for (int k = 0; k < NDIM; ++k) {
    const float ak = fadd(fabsf(Ut[1 + k].h), floor_u);
    as = k == 0 ? ak : fadd(as, ak);
    am = k == 0 ? ak : fmaxf(am, ak);
  }
  const float ua = fmul(R.um, a0);
  const float A = ffma(R.um, ffma(0.5f * NDIM, ua, as), aE);
  const float B = 0.5f * fadd(ua, fadd(fabsf(Ut[1 + DIR].h), floor_u));
  const float W = ffma(0.5f * gm1.h * R.ic.h, A, B), G = fmul(R.ic.h, W);
  const float g = fmul(gm1.h, R.H.h), lim = kRoughLimit * R.c2.h;
  const bool ok = fmul(g, ffma(0.5f, a0, G)) <= fmul(lim, rho_max) &&
                  fmul(g, ffma(0.5f, am, ffma(R.um, G, W))) <= fmul(lim, fmul(amax, rho_max)) &&
                  fmul(g, ffma(0.5f, aE, ffma(R.H.h, G, fmul(R.um, W)))) <= fmul(lim, e_max);
  return !ok;
}
// The corrections to 30 F~ (closed_out with c~ eliminated): T = |u~|^2/2 U~_0 -
// u~.U~_m + U~_E, V = (u~_d U~_0 - U~_d)/2 = c~ B, t = c~ A = (gamma-1)/2 T / c~,
// gs = (sg t + df V) / c~, c~ ngd = df t + sg V.
template <int NDIM, int DIR>
TENO_CERT_HD void closed_df(const teno_df::df (&Ut)[NDIM + 2], const RoeDf<NDIM>& R, const FaceSpeeds& F,
                            teno_df::df gm1, teno_df::df (&o)[NDIM + 2]) {
  using namespace teno_df;
  constexpr int NVAR = NDIM + 2;
  df T = mul(scale(R.q2, 0.5f), Ut[0]);
#pragma unroll
  for (int k = 0; k < NDIM; ++k) T = add(T, neg(mul(R.u[k], Ut[1 + k])));
  T = add(T, Ut[NVAR - 1]);
  const df V = scale(add(mul(R.u[DIR], Ut[0]), neg(Ut[1 + DIR])), 0.5f);
  const df t = mul(mul(df{0.5f * gm1.h, 0.5f * gm1.l}, T), R.ic);
  const df gs = mul(R.ic, add(mul(F.sg, t), mul(F.dd, V)));
  const df cn = add(mul(F.dd, t), mul(F.sg, V));
  o[0] = add(mul(F.amid, Ut[0]), gs);
#pragma unroll
  for (int k = 0; k < NDIM; ++k) {
    o[1 + k] = add(mul(F.amid, Ut[1 + k]), mul(R.u[k], gs));
    if (k == DIR) o[1 + k] = add(o[1 + k], neg(cn));
  }
  o[NVAR - 1] = add(add(mul(F.amid, Ut[NVAR - 1]), mul(R.H, gs)), neg(mul(R.u[DIR], cn)));
}

}  // namespace teno
