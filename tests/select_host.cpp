// select_host.cpp -- test helper: the certified single-precision selection of
// teno_cert.cuh (compiled for the host with -ffp-contract=off, so it rounds
// as on the GPU) behind a C interface for the CPU tests.
#include <cstdint>

#include "teno_cert.cuh"

// e: n x 4 first differences; out[i] = the three delta bits, or -1 where undecided
extern "C" void select_batch(int64_t n, const double* e, float eps4_f, float thr_keep_f, const float* thr_f, int nthr,
                             int b_l, int m_fixed, unsigned keep_all, const float* ct_f, int* out) {
  for (int64_t i = 0; i < n; ++i) {
    const double* w = e + 4 * i;
    unsigned sel = 0;
    out[i] = teno_cert::select_diffs(w[0], w[1], w[2], w[3], eps4_f, thr_keep_f, thr_f, nthr, b_l, m_fixed, keep_all,
                                     ct_f, sel)
                 ? int(sel)
                 : -1;
  }
}
