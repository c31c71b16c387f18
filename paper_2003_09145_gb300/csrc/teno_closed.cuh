// teno_closed.cuh -- the closed form of an interface flux (every stencil kept)
// with its certified test, as the two-pass flux kernels and the batched
// kernel run it: the Roe state and the corrections in two binary32 values
// (teno_df.cuh), U~ and the mass flux in 64-bit fixed point (teno_fixsum.cuh),
// the other fluxes as binary64 chains.
//
// What bounds it: instruction issue (it was FP64 issue: 78 FP64 instructions
// per interface, each holding an SM partition for 64 cycles; now 26 of some
// 2200, the FP64 pipe 45 to 48 % busy, issue 61 to 64 %).  Measured at 256^3 (ms
// per RK3 step): Roe state and corrections in binary64 37.0, in two binary32
// values 28.1, with the cells' binary32 copies from the cell pass (store_planes)
// 25.3, with the certificate's reconstructions in pairs (certify_open2) 24.3,
// with the other passes as they are now 21.3.  Tried on top and dropped: the mass
// flux as a binary64 chain too (slower), the corrections widened and added in two
// FP64 additions instead of one (no gain).
#pragma once

#include "teno_closed_core.cuh"
#include "teno_flux.cuh"

namespace teno {

__device__ __forceinline__ teno_df::df gm1_df(const Scheme& S) { return {S.gm1_h, S.gm1_l}; }

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
// The same from the binary64 arrays, for grids that keep no planes: the values
// that store_planes would have written.
template <int NDIM, int DIR, bool GH, class I>
__device__ __forceinline__ void load_point_d(const double* __restrict__ U, const double* __restrict__ aux,
                                             const GhostCells& gc, int64_t ncell, I c, float (&X)[NDIM + 2], float& u,
                                             float& p) {
#pragma unroll
  for (int v = 0; v < NDIM + 2; ++v) X[v] = near_float(ldc<GH>(U, gc.U, ncell, v, c));
  u = near_float(ldc<GH>(aux, gc.aux, ncell, DIR, c));
  p = near_float(ldc<GH>(aux, gc.aux, ncell, NDIM, c));
}
template <int NDIM, bool GH, class I>
__device__ __forceinline__ RoeCellDf<NDIM> load_roe_cell_d(const double* __restrict__ aux, const GhostCells& gc,
                                                           int64_t ncell, I c) {
  double su[NDIM];
#pragma unroll
  for (int k = 0; k < NDIM; ++k) su[k] = ldc<GH>(aux, gc.aux, ncell, NDIM + 3 + k, c);
  return roe_cell<NDIM>(ldc<GH>(aux, gc.aux, ncell, NDIM + 1, c), ldc<GH>(aux, gc.aux, ncell, NDIM + 2, c), su);
}

// The closed form's Roe state and corrections in binary64, on sums already
// formed (60 U~ and the mass flux in fixed point, the other fluxes): where the
// corrections are not small against the flux scale (closed_df_rough), i.e. at
// shocks.  Out of line, on copies
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
// on the grid path; a3: the halved speeds, F: face_speeds of them.  PF: the cells'
// binary32 values from the planes pf, else converted here.
template <int NDIM, int DIR, bool GH, bool PF = true, class I>
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
  const df gm1 = gm1_df(S);
  RoeDf<NDIM> R;
  {
    RoeCellDf<NDIM> ra, rb;
    if constexpr (PF) {
      ra = load_roe_cell<NDIM, GH>(pf, gc.pf, ncell, cells[2]);
      rb = load_roe_cell<NDIM, GH>(pf, gc.pf, ncell, cells[3]);
    } else {
      ra = load_roe_cell_d<NDIM, GH>(aux, gc, ncell, cells[2]);
      rb = load_roe_cell_d<NDIM, GH>(aux, gc, ncell, cells[3]);
    }
    const float fa = (flips >> 2) & 1u ? -1.0f : 1.0f, fb = (flips >> 3) & 1u ? -1.0f : 1.0f;
    ra.su[DIR] = scale(ra.su[DIR], fa);
    rb.su[DIR] = scale(rb.su[DIR], fb);
    roe_df<NDIM>(ra, rb, gm1, R);
  }
  bool range = F.in_range && roe_df_ok<NDIM>(R, gm1);
  // first pass: the certified test and the largest magnitudes of the summed
  // components (a mirrored point changes signs only)
  unsigned open;
  float xm[NVAR];
  {
    CertIfc<NDIM> C;
    cert_begin_df<NDIM, DIR>(R, F.ha, gm1, C);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      float X[NVAR], u, p;
      if constexpr (PF) load_point_f<NDIM, DIR, GH>(pf, gc.pf, ncell, cells[j], X, u, p);
      else load_point_d<NDIM, DIR, GH>(U, aux, gc, ncell, cells[j], X, u, p);
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
#pragma unroll
    for (int v = 0; v < NVAR; ++v) Ut[v] = from_fixed(AU[v], EU[v]);
    if (!closed_df_rough<NDIM, DIR>(Ut, R, gm1, F.amax, xm[0], xm[NVAR - 1])) {
      df o[NVAR];
      closed_df<NDIM, DIR>(Ut, R, F, gm1, o);
      out[0] = teno_fix::round(AF, EU[1 + DIR] - 1u) + to_double(o[0]);
#pragma unroll
      for (int v = 1; v < NVAR; ++v) out[v] = Fd[v] + to_double(o[v]);
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
