// teno_cert.cuh -- certified single-precision test that a TENO5
// reconstruction keeps every stencil (delta_k = 1 for k = 0, 1, 2 in
// eq. 2.14), for host and device.
//
// GB300's FP64 rate is 1/64 of its FP32 rate, so the flux passes first ask
// FP32 whether the binary64 evaluation would keep every stencil, and only
// evaluate the indicators in binary64 when FP32 cannot prove it.  A test
// here passes only if, for the exact values x_j that the FP32 inputs
// approximate, the scaled indicators (4 beta_k of eq. 2.9-2.11, 4 tau_5 of
// eq. 2.12) satisfy
//     tau_5(x) <= thr * (min_k beta_k(x) + eps) * (1 - 1e-5 + 8 u),
// where thr is the threshold below which the cutoff keeps every stencil
// (Scheme::thr_keep_f).  The margin of about 1e-5 is 2^28 times the rounding
// of a binary64 evaluation of the same quantities (whose errors are at most
// 2^-28 of the FP32 bounds below), so the binary64 decision -- the GPU's and
// the oracle's -- is "keep every stencil" whenever a test passes.
//
// Every FP32 operation is written with its rounding explicit (fadd, fsub,
// fmul, ffma: round to nearest, no contraction), so that the host build (used
// by the CPU tests, compiled with -ffp-contract=off) evaluates bit for bit
// what the device evaluates.  u = 2^-24 is the FP32 unit roundoff.
#pragma once

#include <math.h>

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define TENO_CERT_HD __host__ __device__ __forceinline__
#else
#define TENO_CERT_HD inline
#endif

namespace teno_cert {

TENO_CERT_HD float fadd(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
TENO_CERT_HD float fsub(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fsub_rn(a, b);
#else
  return a - b;
#endif
}
TENO_CERT_HD float fmul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
TENO_CERT_HD float ffma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return std::fmaf(a, b, c);
#endif
}
// fabsf, fminf, fmaxf (exact; NaN-ignoring min/max on both sides) are the
// C library's on the host and CUDA's on the device.

// binary32 approximation of a double built from its high word with integer
// operations only: exponent rebiased, mantissa truncated to 20 bits, so
// |f| <= |x| and |f - x| < 2^-20 |x| for 2^-126 <= |x| < 2^128.  Smaller
// magnitudes become 2^-126 (error below 2^-126); larger ones, infinities and
// NaN become the largest value below 2^128 (their squares overflow, so no
// test below can pass on them).
TENO_CERT_HD float hi_float(double x) {
#ifdef __CUDA_ARCH__
  const unsigned hi = static_cast<unsigned>(__double2hiint(x));
#else
  uint64_t b;
  std::memcpy(&b, &x, sizeof(b));
  const unsigned hi = static_cast<unsigned>(b >> 32);
#endif
  unsigned mag = hi & 0x7fffffffu;
  mag = mag < (897u << 20) ? (897u << 20) : mag;
  mag = mag > ((1150u << 20) | 0xFFFFFu) ? ((1150u << 20) | 0xFFFFFu) : mag;
  const unsigned bits = ((mag - (896u << 20)) << 3) | (hi & 0x80000000u);
#ifdef __CUDA_ARCH__
  return __uint_as_float(bits);
#else
  float f;
  std::memcpy(&f, &bits, sizeof(f));
  return f;
#endif
}

// ---------------------------------------------------------------------------
// certify_keep: v0..v4 are FP32 values with |v_j - x_j| <= r, the test is
// given d with
//     d >= (1 + 2^-19) (r + 2 u W),   d >= 2^-21 W,   W = max |v_j|.
//
// Error budget:
//  * first differences e_k = v_{k+1} - v_k: |e| <= 2W, so each rounds by at
//    most 2uW and |e^ - e(x)| <= 2 r + 2uW;
//  * a_0 = e_1 - e_0 (|.| <= 4W, rounding 4uW) and c_0 = 3 e_1 - e_0 (one
//    rounding, |.| <= 8W): |a^ - a(x)| <= 4 (r + 2uW), |c^ - c(x)| <=
//    8 (r + 2uW); likewise a_1, a_2, c_1, c_2.  Hence |da| <= 4 d and
//    |dc| <= 8 d;
//  * 4 beta = (13/3) a^2 + c^2 from a^, c^ differs from its value at (a, c)
//    by at most (13/3)(2|a^| + 4d) 4d + (2|c^| + 8d) 8d, and its own FP32
//    evaluation (13/3 rounded, one product, one fma) by at most 3.02 u beta^:
//    4 u beta^ is charged;
//  * the (at most six) roundings of each error bound's own evaluation are
//    covered by the 2^-19 = 32 u of slack in d;
//  * dmin = min beta^ + eps (eps rounded down) is within max_k dbeta_k +
//    u dmin of the exact value; 4 u dmin is charged, which also covers the
//    rounding of that sum;
//  * the final comparison's own roundings (a few u) sit inside the 1e-5
//    margin;
//  * an overflow anywhere implies W > 2^125, so d > 2^104 and (4d)^2
//    overflows: dtau is then infinite or NaN and the test fails.
// ---------------------------------------------------------------------------
TENO_CERT_HD bool certify_keep(float v0, float v1, float v2, float v3, float v4, float d, float thr_f,
                               float eps4_f) {
  const float u = 0x1p-24f;
  const float e0 = fsub(v1, v0), e1 = fsub(v2, v1), e2 = fsub(v3, v2), e3 = fsub(v4, v3);
  const float a0 = fsub(e1, e0), a1 = fsub(e2, e1), a2 = fsub(e3, e2);
  const float c0 = ffma(3.0f, e1, -e0), c1 = fadd(e1, e2), c2 = ffma(-3.0f, e2, e3);
  const float k = 13.0f / 3.0f;
  const float b0 = ffma(fmul(k, a0), a0, fmul(c0, c0));
  const float b1 = ffma(fmul(k, a1), a1, fmul(c1, c1));
  const float b2 = ffma(fmul(k, a2), a2, fmul(c2, c2));
  const float da = 4.0f * d, dc = 8.0f * d;   // exact scalings
  // one bound for the three indicators, from the largest |a|, |c| and b (the
  // bound is monotone in them)
  const float am = fmaxf(fabsf(a0), fmaxf(fabsf(a1), fabsf(a2)));
  const float cm = fmaxf(fabsf(c0), fmaxf(fabsf(c1), fabsf(c2)));
  const float db = ffma(4.0f * u, fmaxf(b0, fmaxf(b1, b2)),
                        ffma(fmul(k, ffma(2.0f, am, da)), da, fmul(ffma(2.0f, cm, dc), dc)));
  const float tau = fabsf(fsub(b2, b0));
  const float dtau = ffma(u, tau, fadd(db, db));
  const float dmin = fadd(fminf(b0, fminf(b1, b2)), eps4_f);
  const float ddmin = ffma(4.0f * u, dmin, db);
  return (dtau <= 1.0e38f) && (fadd(tau, dtau) <= fmul(thr_f, fmul(fsub(dmin, ddmin), 1.0f - 1e-5f)));
}

// certify_keep of two reconstructions at once (x and y: the same operations
// in the same order, so the same outcomes), with two operations per
// instruction where the hardware pairs them: bit 0 set where x is not proven
// kept, bit 1 where y is not.
// (On the host a test supplies float2 and the paired operations.)
#if defined(__CUDACC__) || defined(TENO_CERT_PAIRS)
#ifdef __CUDACC__
__device__ __forceinline__
#else
inline
#endif
unsigned certify_open2(float2 v0, float2 v1, float2 v2, float2 v3, float2 v4, float2 d,
                                                  float thr_f, float eps4_f) {
  const float u = 0x1p-24f, k = 13.0f / 3.0f;
  const float2 m1 = make_float2(-1.0f, -1.0f), two = make_float2(2.0f, 2.0f), kk = make_float2(k, k);
  const float2 p3 = make_float2(3.0f, 3.0f), n3 = make_float2(-3.0f, -3.0f);
  // x - y is exact as fma(y, -1, x)
  const float2 e0 = __ffma2_rn(v0, m1, v1), e1 = __ffma2_rn(v1, m1, v2), e2 = __ffma2_rn(v2, m1, v3),
               e3 = __ffma2_rn(v3, m1, v4);
  const float2 a0 = __ffma2_rn(e0, m1, e1), a1 = __ffma2_rn(e1, m1, e2), a2 = __ffma2_rn(e2, m1, e3);
  const float2 ne0 = make_float2(-e0.x, -e0.y);
  const float2 c0 = __ffma2_rn(p3, e1, ne0), c1 = __fadd2_rn(e1, e2), c2 = __ffma2_rn(n3, e2, e3);
  const float2 b0 = __ffma2_rn(__fmul2_rn(kk, a0), a0, __fmul2_rn(c0, c0));
  const float2 b1 = __ffma2_rn(__fmul2_rn(kk, a1), a1, __fmul2_rn(c1, c1));
  const float2 b2 = __ffma2_rn(__fmul2_rn(kk, a2), a2, __fmul2_rn(c2, c2));
  const float2 da = __fmul2_rn(d, make_float2(4.0f, 4.0f)), dc = __fmul2_rn(d, make_float2(8.0f, 8.0f));
  const float2 am = make_float2(fmaxf(fabsf(a0.x), fmaxf(fabsf(a1.x), fabsf(a2.x))),
                                fmaxf(fabsf(a0.y), fmaxf(fabsf(a1.y), fabsf(a2.y))));
  const float2 cm = make_float2(fmaxf(fabsf(c0.x), fmaxf(fabsf(c1.x), fabsf(c2.x))),
                                fmaxf(fabsf(c0.y), fmaxf(fabsf(c1.y), fabsf(c2.y))));
  const float2 bm = make_float2(fmaxf(b0.x, fmaxf(b1.x, b2.x)), fmaxf(b0.y, fmaxf(b1.y, b2.y)));
  const float2 bn = make_float2(fminf(b0.x, fminf(b1.x, b2.x)), fminf(b0.y, fminf(b1.y, b2.y)));
  const float2 db = __ffma2_rn(make_float2(4.0f * u, 4.0f * u), bm,
                               __ffma2_rn(__fmul2_rn(kk, __ffma2_rn(two, am, da)), da,
                                          __fmul2_rn(__ffma2_rn(two, cm, dc), dc)));
  const float2 df = __ffma2_rn(b0, m1, b2);
  const float2 tau = make_float2(fabsf(df.x), fabsf(df.y));
  const float2 dtau = __ffma2_rn(make_float2(u, u), tau, __fadd2_rn(db, db));
  const float2 dmin = __fadd2_rn(bn, make_float2(eps4_f, eps4_f));
  const float2 ddmin = __ffma2_rn(make_float2(4.0f * u, 4.0f * u), dmin, db);
  const float2 lhs = __fadd2_rn(tau, dtau);
  const float2 rhs = __fmul2_rn(make_float2(thr_f, thr_f),
                                __fmul2_rn(__ffma2_rn(ddmin, m1, dmin), make_float2(1.0f - 1e-5f, 1.0f - 1e-5f)));
  const bool kx = dtau.x <= 1.0e38f && lhs.x <= rhs.x, ky = dtau.y <= 1.0e38f && lhs.y <= rhs.y;
  return (kx ? 0u : 1u) | (ky ? 0u : 2u);
}
#endif

// The same test on five binary64 values (one scalar reconstruction),
// truncated by hi_float: |g_j - v_j| <= 2^-20 |v_j| + 2^-126 and
// |v_j| <= |g_j| (1 + 2^-19), so r + 2uW <= 0x1.2p-20 W + 2^-126 (plus
// terms of order 2^-39 W); d = 0x1.3p-20 W + 2^-125 leaves more than 5 %
// of slack, which covers 2^-19 and the rounding of d itself.
TENO_CERT_HD bool certify_keep_values(double v0, double v1, double v2, double v3, double v4, float thr_f,
                                      float eps4_f) {
  const float g0 = hi_float(v0), g1 = hi_float(v1), g2 = hi_float(v2), g3 = hi_float(v3), g4 = hi_float(v4);
  const float W = fmaxf(fmaxf(fmaxf(fabsf(g0), fabsf(g1)), fmaxf(fabsf(g2), fabsf(g3))), fabsf(g4));
  return certify_keep(g0, g1, g2, g3, g4, ffma(0x1.3p-20f, W, 0x1p-125f), thr_f, eps4_f);
}

// ---------------------------------------------------------------------------
// The selections of one reconstruction (LAD, eq. 3.1-3.4, or a fixed C_T) in
// single precision, from the binary64 first differences e_k = v_{k+1} - v_k:
// returns true with the three delta bits in `sel` if the binary64 evaluation
// of the same differences takes them, false if a decision lies within its
// error bound (the caller then decides in binary64).
//
// The differences are truncated to FP32 (error below 2^-20 |e_k| + 2^-126),
// so the bounds scale with the local variation, not with the values.  With
// E_k the larger magnitude of stencil k's two differences, |a_k| <= 2 E_k
// and |c_k| <= 4 E_k are within 2 (2^-20 E_k) + 2u E_k and 4 (2^-20 E_k) + 4u
// E_k of their exact values (c_0, c_2: one rounding each; c_1, a_k too):
// da = 2.2 2^-20 E_k + 2^-123, dc = 2 da cover them.  Then, as in
// certify_keep, db_k bounds |b_k - beta_k| (4u b_k for b_k's own
// evaluation; the slack of da covers the bound's own roundings), dtau bounds
// |tau - tau(e)|, and with D_k = b_k + eps:
//  * D_k is within db_k + 4u D_k of its exact value;
//  * threshold j of m (eq. 3.1) is certainly met when tau + dtau <=
//    thr_j dmin_lo (1 - 1e-6), certainly not when tau - dtau > thr_j dmin_hi
//    (1 + 1e-6), dmin_lo and dmin_hi the least lower and upper bound of the
//    D_k; m is certain when both counts agree; below the keep-all threshold
//    thr_keep every stencil is kept whatever m is;
//  * gamma_k ~ x_k^6 with x_k = 1 + tau / D_k: x_k is within
//    e_k = dtau / (D_k + tau) + db_k / D_k + 12u of its exact value, relative
//    (e the largest of the three); q_k = x_k / max x lies in (0, 1], q_k^6 and
//    its share of the sum of the three are within (1 + e)^24 - 1 <= 26 e
//    (e <= 2^-9) and some 40 roundings (2e-5 >= 335 u) of theirs;
//  * the margins are 2^28 times the binary64 evaluation's rounding.
// m_fixed: the magnitude of C_T; -1: LAD's m; -2: not known here (keep-all only).
// ---------------------------------------------------------------------------
TENO_CERT_HD float fdiv(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fdiv_rn(a, b);
#else
  return a / b;
#endif
}

TENO_CERT_HD bool select_diffs(double f0, double f1, double f2, double f3, float eps4_f, float thr_keep_f,
                               const float* thr_f, int nthr, int b_l, int m_fixed, unsigned keep_all,
                               const float* ct_f, unsigned& sel) {
  const float u = 0x1p-24f;
  const float e0 = hi_float(f0), e1 = hi_float(f1), e2 = hi_float(f2), e3 = hi_float(f3);
  const float a0 = fsub(e1, e0), a1 = fsub(e2, e1), a2 = fsub(e3, e2);
  const float c0 = ffma(3.0f, e1, -e0), c1 = fadd(e1, e2), c2 = ffma(-3.0f, e2, e3);
  const float k = 13.0f / 3.0f;
  const float b0 = ffma(fmul(k, a0), a0, fmul(c0, c0));
  const float b1 = ffma(fmul(k, a1), a1, fmul(c1, c1));
  const float b2 = ffma(fmul(k, a2), a2, fmul(c2, c2));
  const float q = 2.2f * 0x1p-20f, q0 = 0x1p-123f;
  const float da0 = ffma(q, fmaxf(fabsf(e0), fabsf(e1)), q0), da1 = ffma(q, fmaxf(fabsf(e1), fabsf(e2)), q0),
              da2 = ffma(q, fmaxf(fabsf(e2), fabsf(e3)), q0);
  const float dc0 = 2.0f * da0, dc1 = 2.0f * da1, dc2 = 2.0f * da2;
  const float db0 = ffma(4.0f * u, b0, ffma(fmul(k, ffma(2.0f, fabsf(a0), da0)), da0, fmul(ffma(2.0f, fabsf(c0), dc0), dc0)));
  const float db1 = ffma(4.0f * u, b1, ffma(fmul(k, ffma(2.0f, fabsf(a1), da1)), da1, fmul(ffma(2.0f, fabsf(c1), dc1), dc1)));
  const float db2 = ffma(4.0f * u, b2, ffma(fmul(k, ffma(2.0f, fabsf(a2), da2)), da2, fmul(ffma(2.0f, fabsf(c2), dc2), dc2)));
  const float tau = fabsf(fsub(b2, b0));
  const float dtau = ffma(u, tau, fadd(db0, db2));
  if (!(dtau <= 1.0e30f)) return false;
  const float D0 = fadd(b0, eps4_f), D1 = fadd(b1, eps4_f), D2 = fadd(b2, eps4_f);
  const float N0 = fadd(D0, tau), N1 = fadd(D1, tau), N2 = fadd(D2, tau);
  const float i0 = fdiv(1.0f, D0), i1 = fdiv(1.0f, D1), i2 = fdiv(1.0f, D2);
  // dtau / N_k <= dtau / (least N_k)
  const float et = fdiv(dtau, fminf(N0, fminf(N1, N2)));
  const float e = ffma(1.0f + 8.0f * u, fadd(et, fmaxf(fmul(db0, i0), fmaxf(fmul(db1, i1), fmul(db2, i2)))), 12.0f * u);
  if (!(e <= 0x1p-9f)) return false;
  const float lo = fmul(fminf(ffma(-4.0f * u, D0, fsub(D0, db0)),
                              fminf(ffma(-4.0f * u, D1, fsub(D1, db1)), ffma(-4.0f * u, D2, fsub(D2, db2)))),
                        1.0f - 1e-6f);
  const float tp = fadd(tau, dtau);
  if (tp <= fmul(thr_keep_f, lo)) {
    sel = 7u;
    return true;
  }
  if (m_fixed < -1) return false;
  int m = m_fixed;
  if (m_fixed < 0) {
    const float hi = fmul(fminf(ffma(4.0f * u, D0, fadd(D0, db0)),
                                fminf(ffma(4.0f * u, D1, fadd(D1, db1)), ffma(4.0f * u, D2, fadd(D2, db2)))),
                          1.0f + 1e-6f);
    const float tm = fsub(tau, dtau);
    int sure = 0, may = 0;   // the thresholds decrease, so the counts are prefixes
    for (int j = 0; j < nthr; ++j) {
      sure += tp <= fmul(thr_f[j], lo) ? 1 : 0;
      may += tm <= fmul(thr_f[j], hi) ? 1 : 0;
    }
    if (sure != may) return false;
    m = b_l + sure;
  }
  if ((keep_all >> m) & 1u) {
    sel = 7u;
    return true;
  }
  const float x0 = fmul(N0, i0), x1 = fmul(N1, i1), x2 = fmul(N2, i2);
  const float xm = fdiv(1.0f, fmaxf(x0, fmaxf(x1, x2)));
  const float y0 = fmul(x0, xm), y1 = fmul(x1, xm), y2 = fmul(x2, xm);
  const float r0 = fmul(y0, y0), r1 = fmul(y1, y1), r2 = fmul(y2, y2);
  const float h0 = fmul(fmul(r0, r0), r0), h1 = fmul(fmul(r1, r1), r1), h2 = fmul(fmul(r2, r2), r2);
  const float lim = fmul(ct_f[m], fadd(fadd(h0, h1), h2));
  const float M = ffma(26.0f, e, 2e-5f);
  const float up = fmul(lim, fadd(1.0f, M)), dn = fmul(lim, fsub(1.0f, M));
  const bool k0 = h0 >= up, k1 = h1 >= up, k2 = h2 >= up;
  if (!(k0 || h0 <= dn) || !(k1 || h1 <= dn) || !(k2 || h2 <= dn)) return false;
  sel = (k0 ? 1u : 0u) | (k1 ? 2u : 0u) | (k2 ? 4u : 0u);
  return true;
}

// ---------------------------------------------------------------------------
// The test for all 2 nvar reconstructions of one Euler interface.
// cert_begin takes the interface's Roe state (u~, b1/2, b2/2, 1/(2c)) and the
// halved Lax-Friedrichs speeds; cert_point takes one stencil point (its state
// U_j and half u_d, p) to FP32 split characteristic values v+-[j] together
// with the FP32 evaluation of the same expressions on absolute values
// (mp, mm: bounds of the terms that enter each value); cert_keep runs
// certify_keep on every field and side.
//
// Each split value is a sum of products of at most four truncated inputs
// (e.g. (u_d/2 + alpha) b1/2 u~_k U_j) through at most nine FP32 roundings,
// so |v32 - v| <= (4 2^-20 + 9 u)(1 + 2^-18) |.|_abs < 4.6 2^-20 |.|_abs,
// |.|_abs being the absolute evaluation (which the FP32 one approximates
// from below by at most the same relative amount).  The absolute evaluation
// is monotone in every input, so cert_open forms it once per interface, from
// the largest magnitudes over the six points, instead of at every point; it
// also bounds max|v| (FP32 rounding is monotone).  Inputs below 2^-100 add
// an absolute error below 2^-90 for any physical scale.  cert_open passes
// d = (8 2^-20 + 8 u) |.|_abs + 2^-90, more than 1.7 times the r + 2 u W that
// certify_keep needs, and at least 2^-21 W.
//
// The grid path's inputs are not truncated but rounded (cert_begin_f): U, u_d/2,
// p/2, u~, alpha and 1/c~ within 1 u, b1/2 within 5 u and b2/2 within 7 u.  The
// longest chain ((u_d/2 + alpha) b1/2 (u~.m - E)) then stays within 20 u, and
// d = 32 u |.|_abs + 2^-90 is 1.45 times the r + 2 u W of 22 u.  The bound matters where the
// variation is small against the values (large pressures): with 8 2^-20 the
// test proved nothing for |.|_abs above about 50, with 32 u about 190.
// ---------------------------------------------------------------------------
template <int NDIM>
struct CertIfc {
  float uf[NDIM], hb1f, hb2f, hicf, b1f, hudf, haf[NDIM + 2];
  float vp32[6][NDIM + 2], vm32[6][NDIM + 2];
  float xm[NDIM + 2], hum, hpm;   // largest |U_v|, |u_d/2|, |p/2| over the points
  float kd;                       // relative bound of the split values' errors
  int dir;                        // sweep direction (a constant once inlined)
};

// From binary32 values of the Roe state (u~, b1/2, b2/2, 1/(2c)) and of the
// halved speeds; kd: kCertRounded for inputs rounded as above, kCertTruncated
// for truncated ones (hi_float).
constexpr float kCertTruncated = 8.0f * 0x1p-20f + 8.0f * 0x1p-24f, kCertRounded = 32.0f * 0x1p-24f;
template <int NDIM, int DIR>
TENO_CERT_HD void cert_begin_f(const float (&u)[NDIM], float hb1, float hb2, float hic, const float (&ha)[NDIM + 2],
                               float kd, CertIfc<NDIM>& C) {
  constexpr int NVAR = NDIM + 2;
  C.kd = kd;
#pragma unroll
  for (int k = 0; k < NDIM; ++k) C.uf[k] = u[k];
  C.hb1f = hb1;
  C.hb2f = hb2;
  C.hicf = hic;
  // b1 = 2 (b1/2) and u_d/2 from the given values (exact scalings: the same
  // relative bound)
  C.b1f = 2.0f * C.hb1f;
  C.hudf = 0.5f * C.uf[DIR];
#pragma unroll
  for (int f = 0; f < NVAR; ++f) {
    C.haf[f] = ha[f];
    C.xm[f] = 0.0f;
  }
  C.hum = C.hpm = 0.0f;
  C.dir = DIR;
}

template <int NDIM, int DIR>
TENO_CERT_HD void cert_begin(const double (&u)[NDIM], double hb1, double hb2, double hic,
                             const double (&alpha)[NDIM + 2], CertIfc<NDIM>& C) {
  float uf[NDIM], ha[NDIM + 2];
#pragma unroll
  for (int k = 0; k < NDIM; ++k) uf[k] = hi_float(u[k]);
#pragma unroll
  for (int f = 0; f < NDIM + 2; ++f) ha[f] = hi_float(alpha[f]);
  cert_begin_f<NDIM, DIR>(uf, hi_float(hb1), hi_float(hb2), hi_float(hic), ha, kCertTruncated, C);
}

// Point j: binary32 values X of U_j (normal momentum already mirrored at a
// wall), of u_d/2 and of p/2.  The split values follow the binary64
// characteristic path: w = L U_j, t = (p/2) z, v+ = (u_d/2 + alpha) w + t,
// v- = v+ - 2 alpha w.
template <int NDIM, int DIR>
TENO_CERT_HD void cert_point_f(int j, const float (&X)[NDIM + 2], float huf, float hpf, CertIfc<NDIM>& C) {
  constexpr int NVAR = NDIM + 2;
#pragma unroll
  for (int v = 0; v < NVAR; ++v) C.xm[v] = fmaxf(C.xm[v], fabsf(X[v]));
  C.hum = fmaxf(C.hum, fabsf(huf));
  C.hpm = fmaxf(C.hpm, fabsf(hpf));
  float Sv = -X[NVAR - 1];
#pragma unroll
  for (int k = 0; k < NDIM; ++k) Sv = ffma(C.uf[k], X[1 + k], Sv);
  const float A = ffma(C.hb2f, X[0], -fmul(C.hb1f, Sv));
  const float B = fmul(ffma(C.uf[DIR], X[0], -X[1 + DIR]), C.hicf);
  float w[NVAR];
  w[0] = fadd(A, B);
  w[1] = ffma(-2.0f, A, X[0]);
  {
    int f = 2;
#pragma unroll
    for (int t = 0; t < NDIM; ++t) {
      if (t == DIR) continue;
      w[f] = ffma(-C.uf[t], X[0], X[1 + t]);
      ++f;
    }
  }
  w[NVAR - 1] = fsub(A, B);
  const float az = fmul(hpf, fmul(C.b1f, fsub(huf, C.hudf)));
  const float bz = fmul(hpf, C.hicf);
#pragma unroll
  for (int f = 0; f < NVAR; ++f) {
    const float t = (f == 0) ? fsub(az, bz) : (f == NVAR - 1) ? fadd(az, bz) : -2.0f * az;
    const float s = fadd(huf, C.haf[f]);
    C.vp32[j][f] = (f >= 2 && f < NVAR - 1) ? fmul(s, w[f]) : ffma(s, w[f], t);
    C.vm32[j][f] = ffma(-2.0f * C.haf[f], w[f], C.vp32[j][f]);
  }
}

template <int NDIM, int DIR>
TENO_CERT_HD void cert_point(int j, const double (&Uj)[NDIM + 2], double unj, double pnj, CertIfc<NDIM>& C) {
  float X[NDIM + 2];
#pragma unroll
  for (int v = 0; v < NDIM + 2; ++v) X[v] = hi_float(Uj[v]);
  cert_point_f<NDIM, DIR>(j, X, hi_float(unj), hi_float(pnj), C);
}

// cert_open: bit 2 f (side v+) and 2 f + 1 (side v-) set where the test does
// not prove that field f keeps every stencil; cert_keep: none is set.
template <int NDIM>
TENO_CERT_HD unsigned cert_open(const CertIfc<NDIM>& C, float thr_f, float eps4_f) {
  constexpr int NVAR = NDIM + 2;
  // the absolute evaluation of cert_point_f's expressions at the maxima
  float Sa = C.xm[NVAR - 1];
#pragma unroll
  for (int k = 0; k < NDIM; ++k) Sa = ffma(fabsf(C.uf[k]), C.xm[1 + k], Sa);
  const float Aa = ffma(fabsf(C.hb2f), C.xm[0], fmul(fabsf(C.hb1f), Sa));
  const float Ba = fmul(ffma(fabsf(C.uf[C.dir]), C.xm[0], C.xm[1 + C.dir]), fabsf(C.hicf));
  float wa[NVAR];
  wa[0] = wa[NVAR - 1] = fadd(Aa, Ba);
  wa[1] = ffma(2.0f, Aa, C.xm[0]);
  {
    int f = 2;
#pragma unroll
    for (int t = 0; t < NDIM; ++t) {
      if (t == C.dir) continue;
      wa[f] = ffma(fabsf(C.uf[t]), C.xm[0], C.xm[1 + t]);
      ++f;
    }
  }
  const float aza = fmul(C.hpm, fmul(fabsf(C.b1f), fadd(C.hum, fabsf(C.hudf))));
  const float bza = fmul(C.hpm, fabsf(C.hicf));
  const float kd = C.kd;
  unsigned open = 0u;
#pragma unroll
  for (int f = 0; f < NVAR; ++f) {
    const float ta = (f == 0 || f == NVAR - 1) ? fadd(aza, bza) : (f == 1) ? 2.0f * aza : 0.0f;
    const float mp = ffma(fadd(C.hum, C.haf[f]), wa[f], ta);
    const float mm = ffma(2.0f * C.haf[f], wa[f], mp);
#ifdef __CUDA_ARCH__
    open |= certify_open2(make_float2(C.vp32[0][f], C.vm32[5][f]), make_float2(C.vp32[1][f], C.vm32[4][f]),
                          make_float2(C.vp32[2][f], C.vm32[3][f]), make_float2(C.vp32[3][f], C.vm32[2][f]),
                          make_float2(C.vp32[4][f], C.vm32[1][f]),
                          make_float2(ffma(kd, mp, 0x1p-90f), ffma(kd, mm, 0x1p-90f)), thr_f, eps4_f)
            << (2 * f);
#else
    if (!certify_keep(C.vp32[0][f], C.vp32[1][f], C.vp32[2][f], C.vp32[3][f], C.vp32[4][f],
                      ffma(kd, mp, 0x1p-90f), thr_f, eps4_f))
      open |= 1u << (2 * f);
    if (!certify_keep(C.vm32[5][f], C.vm32[4][f], C.vm32[3][f], C.vm32[2][f], C.vm32[1][f],
                      ffma(kd, mm, 0x1p-90f), thr_f, eps4_f))
      open |= 2u << (2 * f);
#endif
  }
  return open;
}

template <int NDIM>
TENO_CERT_HD bool cert_keep(const CertIfc<NDIM>& C, float thr_f, float eps4_f) {
  return cert_open<NDIM>(C, thr_f, eps4_f) == 0u;
}

}  // namespace teno_cert
