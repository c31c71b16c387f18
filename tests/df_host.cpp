// df_host.cpp -- test helper: teno_df.cuh (compiled for the host with
// -ffp-contract=off, so every operation rounds as on the GPU, its two seeds
// apart) behind a C interface for the CPU tests.
#include <cstdint>

#include "teno_df.cuh"

using teno_df::df;

// op: 0 from_double, 1 add, 2 mul, 3 recip, 4 rsqrt, 5 to_double(from_double),
// 6 sqr; a, b doubles; out[3 i] = h, l (as doubles), and to_double's value
extern "C" void df_batch(int op, int64_t n, const double* a, const double* b, double* out) {
  for (int64_t i = 0; i < n; ++i) {
    const df x = teno_df::from_double(a[i]), y = teno_df::from_double(b[i]);
    df r = x;
    if (op == 1) r = teno_df::add(x, y);
    if (op == 2) r = teno_df::mul(x, y);
    if (op == 3) r = teno_df::recip(x);
    if (op == 4) r = teno_df::rsqrt(x);
    if (op == 6) r = teno_df::sqr(x);
    out[3 * i] = r.h;
    out[3 * i + 1] = r.l;
    out[3 * i + 2] = teno_df::to_double(r);
  }
}

extern "C" void df_fixed(int64_t n, const int64_t* A, const uint32_t* E, double* out) {
  for (int64_t i = 0; i < n; ++i) {
    const df r = teno_df::from_fixed(A[i], E[i]);
    out[2 * i] = r.h;
    out[2 * i + 1] = r.l;
  }
}
