// closed_host.cpp -- test helper: the closed form's two-binary32 arithmetic
// (teno_closed_core.cuh, compiled for the host with -ffp-contract=off, so every
// operation rounds as on the GPU, the two seeds apart) behind a C interface for
// the CPU tests.
#include <cstdint>
#include <cstring>

// the seeds, off by as many ulps as the hardware's may be
static int g_seed_ulps = 0;
static inline float perturbed(float y, int most);
#define TENO_HOST_SEED(y, most) perturbed(y, most)
#include "teno_closed_core.cuh"

static inline float perturbed(float y, int most) {
  const int d = g_seed_ulps < -most ? -most : (g_seed_ulps > most ? most : g_seed_ulps);
  return teno_df::from_bits(teno_df::bits(y) + d);
}

extern "C" void closed_seed_ulps(int n) { g_seed_ulps = n; }

namespace {

using teno_df::df;

// One interface: states U[6][nvar], u_d/2 and p/2 [6], the Roe cells' sqrt(rho),
// (E+p)/sqrt(rho), m/sqrt(rho) (two each) and the halved speeds.  out: [0] in range,
// [1] rough, [2] open mask, then the corrections to 30 F~ [nvar]; A, E: the sums
// 60 U~ = A 2^(E - 1078).
template <int NDIM, int DIR>
void one(const double* U, const double* un, const double* pn, const double* sr, const double* sh, const double* su,
         const double* a, double gm1, float thr_f, float eps4_f, double* out, int64_t* A, uint32_t* E) {
  constexpr int NVAR = NDIM + 2;
  const float gh = static_cast<float>(gm1);
  const df g{gh, static_cast<float>(gm1 - static_cast<double>(gh))};
  const double a3[3] = {a[0], a[1], a[2]};
  const teno::FaceSpeeds F = teno::face_speeds(a3);
  double s2[NDIM], s3[NDIM];
  for (int k = 0; k < NDIM; ++k) s2[k] = su[k], s3[k] = su[NDIM + k];
  teno::RoeDf<NDIM> R;
  teno::roe_df<NDIM>(teno::roe_cell<NDIM>(sr[0], sh[0], s2), teno::roe_cell<NDIM>(sr[1], sh[1], s3), g, R);
  teno::CertIfc<NDIM> C;
  teno::cert_begin_df<NDIM, DIR>(R, F.ha, g, C);
  for (int j = 0; j < 6; ++j) {
    float X[NVAR];
    for (int v = 0; v < NVAR; ++v) X[v] = teno::near_float(U[j * NVAR + v]);
    teno_cert::cert_point_f<NDIM, DIR>(j, X, teno::near_float(un[j]), teno::near_float(pn[j]), C);
  }
  const bool range = F.in_range && teno::roe_df_ok<NDIM>(R, g) && teno::df_range(C.xm[0], C.xm[NVAR - 1]);
  constexpr int kM[6] = {1, -5, 10, -10, 5, -1};
  df Ut[NVAR], o[NVAR];
  for (int v = 0; v < NVAR; ++v) {
    E[v] = (teno_df::bits(C.xm[v]) >> 23) + 896u;
    A[v] = 0;
    for (int j = 0; j < 6; ++j) A[v] += kM[j] * teno_fix::term(U[j * NVAR + v], E[v]);
    Ut[v] = teno_df::from_fixed(A[v], E[v]);
  }
  out[0] = range;
  out[1] = range && teno::closed_df_rough<NDIM, DIR>(Ut, R, g, F.amax, C.xm[0], C.xm[NVAR - 1]);
  out[2] = range ? teno_cert::cert_open<NDIM>(C, thr_f, eps4_f) : 0;
  teno::closed_df<NDIM, DIR>(Ut, R, F, g, o);
  for (int v = 0; v < NVAR; ++v) out[3 + v] = teno_df::to_double(o[v]);
}

}  // namespace

extern "C" void closed_batch(int ndim, int dir, int64_t n, const double* U, const double* un, const double* pn,
                             const double* sr, const double* sh, const double* su, const double* a, double gm1,
                             float thr_f, float eps4_f, double* out, int64_t* A, uint32_t* E) {
  const int nv = ndim + 2;
  for (int64_t i = 0; i < n; ++i) {
    auto go = [&](auto f) {
      f(U + i * 6 * nv, un + 6 * i, pn + 6 * i, sr + 2 * i, sh + 2 * i, su + 2 * ndim * i, a + 3 * i, gm1, thr_f, eps4_f,
        out + i * (3 + nv), A + i * nv, E + i * nv);
    };
    if (ndim == 1) go(one<1, 0>);
    else if (ndim == 2) dir == 0 ? go(one<2, 0>) : go(one<2, 1>);
    else dir == 0 ? go(one<3, 0>) : (dir == 1 ? go(one<3, 1>) : go(one<3, 2>));
  }
}
