// teno_closed.cuh -- the closed form of an interface flux (every stencil kept)
// with its certified test, as the two-pass flux kernels and the batched
// kernel run it: the Roe state and the corrections in two binary32 values
// (teno_df.cuh), U~ and the mass flux in 64-bit fixed point (teno_fixsum.cuh),
// the other fluxes as binary64 chains.
//
// What bounds it: instruction issue (it was FP64 issue: 78 FP64 instructions
// per interface, each holding an SM partition for 64 cycles; now 29, the FP64
// pipe 40 % busy).  Measured at 256^3 (ms per RK3 step): Roe state and
// corrections in binary64 37.0, in two binary32 values 28.1, with the cells'
// binary32 copies from the cell pass (store_planes) 25.3, with the
// certificate's reconstructions in pairs (certify_open2) 24.3.  Tried on top
// and dropped: the mass flux as a binary64 chain too (slower), the corrections
// widened and added in two FP64 additions instead of one (no gain).
#pragma once

#include "teno_df.cuh"
#include "teno_flux.cuh"

namespace teno {

// x rounded to binary32 (within 2^-24 and a bit, relative) by integer and FP32
// operations, for 2^-100 <= |x| < 2^100; beyond that hi_float's clamped
// truncation
__device__ __forceinline__ float near_float(double x) {
  const uint32_t e = (teno_fix::hi_word(x) >> 20) & 0x7FFu;
  if (e - 923u >= 200u) return hi_float(x);
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
__device__ __forceinline__ FaceSpeeds face_speeds(const double (&a3)[3]) {
  using namespace teno_df;
  FaceSpeeds F;
  const df am = from_double(a3[0]), a0 = from_double(a3[1]), ap = from_double(a3[2]);
  const df d0 = add(am, neg(a0)), dE = add(ap, neg(a0));
  F.amid = a0;
  F.sg = add(d0, dE);
  F.dd = add(d0, neg(dE));
#pragma unroll
  for (int s = 0; s < 3; ++s) F.ha[s] = near_float(a3[s]);
  F.amax = 2.0f * fmaxf(F.ha[0], F.ha[2]);
  F.in_range = F.amax >= 0x1p-19f && F.amax <= 0x1p30f;
  return F;
}

// What the closed form's first pass and its Roe state read of a cell, in
// binary32, written once per cell by the cell pass (converting it at each of
// the eighteen stencil points that read the cell took some 280 instructions
// per interface): planes of float4, pf[plane_count(NDIM)][ncell].  Rounded
// values of U, p/2 and u_k/2 (near_float), and sqrt(rho), (E+p)/sqrt(rho),
// m_k/sqrt(rho) as two binary32 values (from_double):
//   1D: {rho, m, E, p/2}, {u/2, 0, su}, {sr, sh}
//   2D: {rho, m_0, m_1, E}, {p/2, u_0/2, u_1/2, 0}, {sr, sh}, {su_0, su_1}
//   3D: {rho, m_0, m_1, m_2}, {E, p/2, u_0/2, u_1/2}, {u_2/2, 0, su_2}, {sr, sh}, {su_0, su_1}
template <int NDIM>
__device__ __forceinline__ void store_planes(float4* __restrict__ pf, int64_t ncell, int64_t c,
                                             const double (&U)[NDIM + 2], const double (&uh)[NDIM], double ph, double sr,
                                             double sh, const double (&su)[NDIM]) {
  using namespace teno_df;
  float X[NDIM + 2], u[NDIM];
#pragma unroll
  for (int v = 0; v < NDIM + 2; ++v) X[v] = near_float(U[v]);
#pragma unroll
  for (int k = 0; k < NDIM; ++k) u[k] = near_float(uh[k]);
  const float p = near_float(ph);
  const df r = from_double(sr), h = from_double(sh), s0 = from_double(su[0]);
  float4* o = pf + c;
  if constexpr (NDIM == 1) {
    o[0] = make_float4(X[0], X[1], X[2], p);
    o[ncell] = make_float4(u[0], 0.0f, s0.h, s0.l);
    o[2 * ncell] = make_float4(r.h, r.l, h.h, h.l);
  } else if constexpr (NDIM == 2) {
    const df s1 = from_double(su[1]);
    o[0] = make_float4(X[0], X[1], X[2], X[3]);
    o[ncell] = make_float4(p, u[0], u[1], 0.0f);
    o[2 * ncell] = make_float4(r.h, r.l, h.h, h.l);
    o[3 * ncell] = make_float4(s0.h, s0.l, s1.h, s1.l);
  } else {
    const df s1 = from_double(su[1]), s2 = from_double(su[2]);
    o[0] = make_float4(X[0], X[1], X[2], X[3]);
    o[ncell] = make_float4(X[4], p, u[0], u[1]);
    o[2 * ncell] = make_float4(u[2], 0.0f, s2.h, s2.l);
    o[3 * ncell] = make_float4(r.h, r.l, h.h, h.l);
    o[4 * ncell] = make_float4(s0.h, s0.l, s1.h, s1.l);
  }
}

// plane k of cell c, or of the ghost block when GH and c is a virtual cell
template <bool GH, class I>
__device__ __forceinline__ const float4* plane(const float4* __restrict__ pf, const float4* __restrict__ gpf,
                                               int64_t ncell, int k, I c) {
  if (GH && (int64_t)c >= ncell) return gpf + k * kGhostSlots + ((int64_t)c - ncell);
  return pf + k * ncell + c;
}

// U, u_DIR/2 and p/2 of cell c
template <int NDIM, int DIR, bool GH, class I>
__device__ __forceinline__ void load_point_f(const float4* __restrict__ pf, const float4* __restrict__ gpf,
                                             int64_t ncell, I c, float (&X)[NDIM + 2], float& u, float& p) {
  const float4 a = *plane<GH>(pf, gpf, ncell, 0, c);
  if constexpr (NDIM == 1) {
    X[0] = a.x, X[1] = a.y, X[2] = a.z, p = a.w;
    u = plane<GH>(pf, gpf, ncell, 1, c)->x;
  } else {
    const float4 b = *plane<GH>(pf, gpf, ncell, 1, c);
    X[0] = a.x, X[1] = a.y, X[2] = a.z, X[3] = a.w;
    if constexpr (NDIM == 2) {
      p = b.x;
      u = DIR == 0 ? b.y : b.z;
    } else {
      X[4] = b.x;
      p = b.y;
      if constexpr (DIR == 2) u = plane<GH>(pf, gpf, ncell, 2, c)->x;
      else u = DIR == 0 ? b.z : b.w;
    }
  }
}

// The Roe state in two binary32 values, from the cells' sqrt(rho),
// (E+p)/sqrt(rho) and m_k/sqrt(rho) (roe_interface's average): u~, |u~|^2, H~,
// c~^2 and 1/c~.
template <int NDIM>
struct RoeDf {
  teno_df::df u[NDIM], q2, H, c2, ic;
};
template <int NDIM>
struct RoeCellDf {   // one cell's contribution
  teno_df::df sr, sh, su[NDIM];
};
template <int NDIM, bool GH, class I>
__device__ __forceinline__ RoeCellDf<NDIM> load_roe_cell(const float4* __restrict__ pf, const float4* __restrict__ gpf,
                                                         int64_t ncell, I c) {
  RoeCellDf<NDIM> R;
  const float4 d = *plane<GH>(pf, gpf, ncell, NDIM == 3 ? 3 : 2, c);
  R.sr = {d.x, d.y};
  R.sh = {d.z, d.w};
  if constexpr (NDIM == 1) {
    const float4 e = *plane<GH>(pf, gpf, ncell, 1, c);
    R.su[0] = {e.z, e.w};
  } else {
    const float4 e = *plane<GH>(pf, gpf, ncell, NDIM == 3 ? 4 : 3, c);
    R.su[0] = {e.x, e.y};
    R.su[1] = {e.z, e.w};
    if constexpr (NDIM == 3) {
      const float4 f = *plane<GH>(pf, gpf, ncell, 2, c);
      R.su[2] = {f.z, f.w};
    }
  }
  return R;
}
template <int NDIM>
__device__ __forceinline__ RoeCellDf<NDIM> roe_cell(double sr, double sh, const double (&su)[NDIM]) {
  RoeCellDf<NDIM> R;
  R.sr = teno_df::from_double(sr);
  R.sh = teno_df::from_double(sh);
#pragma unroll
  for (int k = 0; k < NDIM; ++k) R.su[k] = teno_df::from_double(su[k]);
  return R;
}
template <int NDIM>
__device__ __forceinline__ void roe_df(const RoeCellDf<NDIM>& a, const RoeCellDf<NDIM>& b, const Scheme& S,
                                       RoeDf<NDIM>& R) {
  using namespace teno_df;
  const df y = recip(add(a.sr, b.sr));
#pragma unroll
  for (int k = 0; k < NDIM; ++k) {
    R.u[k] = mul(add(a.su[k], b.su[k]), y);
    R.q2 = k == 0 ? sqr(R.u[0]) : add(R.q2, sqr(R.u[k]));
  }
  R.H = mul(add(a.sh, b.sh), y);
  R.c2 = mul(df{S.gm1_h, S.gm1_l}, add(R.H, scale(R.q2, -0.5f)));
  R.ic = teno_df::rsqrt(R.c2);
}

// The certificate's view of that Roe state, rounded to binary32, where
// roe_df_ok holds, i.e. where c~^2 keeps 2^-6 of (gamma - 1) H~ (Mach numbers
// below about 18 for gamma = 1.4; c~^2 is then good to 2^-38).
template <int NDIM, int DIR>
__device__ __forceinline__ void cert_begin_df(const RoeDf<NDIM>& R, const float (&ha3)[3], const Scheme& S,
                                              CertIfc<NDIM>& C) {
  using teno_cert::fadd;
  using teno_cert::fmul;
  float uf[NDIM], ha[NDIM + 2];
#pragma unroll
  for (int k = 0; k < NDIM; ++k) uf[k] = fadd(R.u[k].h, R.u[k].l);
#pragma unroll
  for (int f = 0; f < NDIM + 2; ++f) ha[f] = ha3[f == 0 ? 0 : (f == NDIM + 1 ? 2 : 1)];
  const float ic = fadd(R.ic.h, R.ic.l);
  const float hb1 = fmul(0.5f * S.gm1_h, fmul(ic, ic));
  teno_cert::cert_begin_f<NDIM, DIR>(uf, hb1, fmul(0.5f * hb1, fadd(R.q2.h, R.q2.l)), 0.5f * ic, ha,
                                     teno_cert::kCertRounded, C);
}
template <int NDIM>
__device__ __forceinline__ bool roe_df_ok(const RoeDf<NDIM>& R, const Scheme& S) {
  return R.c2.h > 0x1p-6f * S.gm1_h * R.H.h;
}

// 2^-20 <= max rho < 2^30 and max E < 2^95 keep every term of the test and of
// teno_df in binary32's range; |u| and c are bounded by the speeds.
__device__ __forceinline__ bool df_range(float rho_max, float e_max) {
  return rho_max >= 0x1p-20f && rho_max < 0x1p30f && e_max < 0x1p95f;
}

// The closed form's Roe state and corrections in binary64, on sums already
// formed (60 U~ and the mass flux in fixed point, the other fluxes): where U~
// is not small against the flux scale, i.e. at shocks.  Out of line, on copies
// of its inputs, so that the common form's values stay in registers.
template <int NDIM>
struct ClosedSums {
  uint32_t EU[NDIM + 2];
  int64_t AU[NDIM + 2], AF;
  double Fd[NDIM + 2];
};
template <int NDIM, int DIR, bool GH, class I>
__device__ __noinline__ void closed_rough(const double* __restrict__ aux, int64_t ncell, I ca, I cb, unsigned flips,
                                          double am, double a0, double ap, const Scheme& S, const ClosedSums<NDIM>& X,
                                          double (&out)[NDIM + 2], int* __restrict__ status, const GhostCells& gc) {
  constexpr int NVAR = NDIM + 2;
  const double a3[3] = {am, a0, ap};
  double alpha[NVAR], nal[NVAR], su2[NDIM], su3[NDIM];
  spread_speeds<NDIM>(a3, alpha, nal);
  RoeIfc<NDIM> R;
#pragma unroll
  for (int k = 0; k < NDIM; ++k) {
    su2[k] = ldc<GH>(aux, gc.aux, ncell, NDIM + 3 + k, ca);
    su3[k] = ldc<GH>(aux, gc.aux, ncell, NDIM + 3 + k, cb);
  }
  su2[DIR] = flip_sign(su2[DIR], (flips >> 2) & 1u);
  su3[DIR] = flip_sign(su3[DIR], (flips >> 3) & 1u);
  roe_interface<NDIM, DIR>(ldc<GH>(aux, gc.aux, ncell, NDIM + 1, ca), ldc<GH>(aux, gc.aux, ncell, NDIM + 1, cb),
                           ldc<GH>(aux, gc.aux, ncell, NDIM + 2, ca), ldc<GH>(aux, gc.aux, ncell, NDIM + 2, cb), su2,
                           su3, S, R, status);
  double Ft[NVAR], Ut[NVAR];
#pragma unroll
  for (int v = 0; v < NVAR; ++v) {
    Ft[v] = v == 0 ? teno_fix::round(X.AF, X.EU[1 + DIR]) : X.Fd[v];
    Ut[v] = teno_fix::round(X.AU[v], X.EU[v]);
  }
  closed_out<NDIM, DIR>(Ft, Ut, R, nal, out);
}

// The flux of one interface with every stencil kept, and the mask of its open
// reconstructions (see interface_flux_closed_wide, which takes over, all in
// binary64, where the interface leaves teno_df's range; closed_rough: near
// shocks).  I: the cell index type, 32 bits
// on the grid path; a3: the halved speeds, F: face_speeds of them.
template <int NDIM, int DIR, bool GH, class I>
__device__ __forceinline__ unsigned interface_flux_closed(const double* __restrict__ U,
                                                          const double* __restrict__ aux,
                                                          const double* __restrict__ fh,
                                                          const float4* __restrict__ pf, int64_t ncell,
                                                          const I (&cells)[6], unsigned flips,
                                                          const double (&a3)[3], const FaceSpeeds& F,
                                                          const Scheme& S, double (&out)[NDIM + 2],
                                                          int* __restrict__ status, const GhostCells& gc) {
  using namespace teno_df;
  constexpr int NVAR = NDIM + 2;
  if (S.keep_idx < 0) return kRough | kAllOpen<NDIM>;
  const double* gfh = GH ? gc.fh + DIR * (NVAR - 1) * kGhostSlots : nullptr;
  RoeDf<NDIM> R;
  {
    RoeCellDf<NDIM> ra = load_roe_cell<NDIM, GH>(pf, gc.pf, ncell, cells[2]);
    RoeCellDf<NDIM> rb = load_roe_cell<NDIM, GH>(pf, gc.pf, ncell, cells[3]);
    const float fa = (flips >> 2) & 1u ? -1.0f : 1.0f, fb = (flips >> 3) & 1u ? -1.0f : 1.0f;
    ra.su[DIR] = scale(ra.su[DIR], fa);
    rb.su[DIR] = scale(rb.su[DIR], fb);
    roe_df<NDIM>(ra, rb, S, R);
  }
  bool range = F.in_range && roe_df_ok<NDIM>(R, S);
  // first pass: the certified test and the largest magnitudes of the summed
  // components (a mirrored point changes signs only)
  unsigned open;
  float xm[NVAR];
  {
    CertIfc<NDIM> C;
    cert_begin_df<NDIM, DIR>(R, F.ha, S, C);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      float X[NVAR], u, p;
      load_point_f<NDIM, DIR, GH>(pf, gc.pf, ncell, cells[j], X, u, p);
      const uint32_t fj = ((flips >> j) & 1u) << 31;
      X[1 + DIR] = __uint_as_float(__float_as_uint(X[1 + DIR]) ^ fj);
      u = __uint_as_float(__float_as_uint(u) ^ fj);
      teno_cert::cert_point_f<NDIM, DIR>(j, X, u, p, C);
    }
    range = range && df_range(C.xm[0], C.xm[NVAR - 1]);
    open = cert_open<NDIM>(C, S);
#pragma unroll
    for (int v = 0; v < NVAR; ++v) xm[v] = C.xm[v];
  }
  if (range) {
    // second pass: 60 U~ and the mass flux in fixed point on the grids of the
    // components' largest exponents, the other fluxes as binary64 chains
    // (see ClosedFix), fully unrolled: the weights are constants (22.1 ms per
    // 256^3 step against 22.5 in two rounds of three and 24.0 rolled).
    constexpr int kC[6] = {1, -8, 37, 37, -8, 1}, kM[6] = {1, -5, 10, -10, 5, -1};
    uint32_t EU[NVAR];
    int64_t AU[NVAR], AF = 0;
    double Fd[NVAR];
#pragma unroll
    for (int v = 0; v < NVAR; ++v) {
      EU[v] = (__float_as_uint(xm[v]) >> 23) + 896u;
      AU[v] = 0;
      Fd[v] = 0.0;
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const I c = cells[j];
      const bool fj = (flips >> j) & 1u;
#pragma unroll
      for (int v = 0; v < NVAR; ++v) {
        const double x = flip_sign(ldc<GH>(U, gc.U, ncell, v, c), fj && v == 1 + DIR);
        const int64_t X = teno_fix::term(x, EU[v]);
        AU[v] += kM[j] * X;
        if (v == 1 + DIR) AF += kC[j] * X;
      }
#pragma unroll
      for (int v = 1; v < NVAR; ++v) {
        const double f = flip_sign(ldc<GH>(fh, gfh, ncell, v - 1, c), fj && v != 1 + DIR);
        if (j == 0) Fd[v] = f;
        else if (j == 5) Fd[v] += f;
        else Fd[v] = fma(double(kC[j]), f, Fd[v]);
      }
    }
    df Ut[NVAR];
    bool rough = false;
    // U~ against the flux scale: |60 U~| <= 60 2^-8 (rho, alpha rho, E),
    // tightened by c~^2 / ((gamma - 1) H~), the digits that c~^2 lost
    const float gH = S.gm1_h * R.H.h, lim = (60.0f * 0x1p-8f) * R.c2.h;
#pragma unroll
    for (int v = 0; v < NVAR; ++v) {
      Ut[v] = from_fixed(AU[v], EU[v]);
      const float sc = v == 0 ? xm[0] : (v == NVAR - 1 ? xm[NVAR - 1] : xm[0] * F.amax);
      rough = rough || !(fabsf(Ut[v].h) * gH <= lim * sc);
    }
    if (!rough) {
      // closed_out with c~ eliminated: T = |u~|^2/2 U~_0 - u~.U~_m + U~_E,
      // V = (u~_d U~_0 - U~_d)/2 = c~ B, t = c~ A = (gamma-1)/2 T / c~,
      // gs = (sg t + df V) / c~, c~ ngd = df t + sg V
      df T = mul(scale(R.q2, 0.5f), Ut[0]);
#pragma unroll
      for (int k = 0; k < NDIM; ++k) T = add(T, neg(mul(R.u[k], Ut[1 + k])));
      T = add(T, Ut[NVAR - 1]);
      const df V = scale(add(mul(R.u[DIR], Ut[0]), neg(Ut[1 + DIR])), 0.5f);
      const df t = mul(mul(df{0.5f * S.gm1_h, 0.5f * S.gm1_l}, T), R.ic);
      const df gs = mul(R.ic, add(mul(F.sg, t), mul(F.dd, V)));
      const df cn = add(mul(F.dd, t), mul(F.sg, V));
      out[0] = teno_fix::round(AF, EU[1 + DIR] - 1u) + to_double(add(mul(F.amid, Ut[0]), gs));
#pragma unroll
      for (int k = 0; k < NDIM; ++k) {
        df o = add(mul(F.amid, Ut[1 + k]), mul(R.u[k], gs));
        if (k == DIR) o = add(o, neg(cn));
        out[1 + k] = Fd[1 + k] + to_double(o);
      }
      out[NVAR - 1] =
          Fd[NVAR - 1] + to_double(add(add(mul(F.amid, Ut[NVAR - 1]), mul(R.H, gs)), neg(mul(R.u[DIR], cn))));
    } else {
      ClosedSums<NDIM> X;
      double o[NVAR];
#pragma unroll
      for (int v = 0; v < NVAR; ++v) {
        X.EU[v] = EU[v];
        X.AU[v] = AU[v];
        X.Fd[v] = Fd[v];
      }
      X.AF = AF;
      closed_rough<NDIM, DIR, GH, I>(aux, ncell, cells[2], cells[3], flips, a3[0], a3[1], a3[2], S, X, o, status, gc);
#pragma unroll
      for (int v = 0; v < NVAR; ++v) out[v] = o[v];
    }
  } else {
    I cc[6];
    double aa[3] = {a3[0], a3[1], a3[2]}, o[NVAR];
#pragma unroll
    for (int j = 0; j < 6; ++j) cc[j] = cells[j];
    open = interface_flux_closed_wide<NDIM, DIR, GH, I>(U, aux, fh, ncell, cc, flips, aa, S, o, status, gc);
#pragma unroll
    for (int v = 0; v < NVAR; ++v) out[v] = o[v];
  }
  return open;
}

}  // namespace teno
