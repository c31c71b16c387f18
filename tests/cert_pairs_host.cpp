// cert_pairs_host.cpp -- test helper: the paired certificate (certify_open2) on the
// host, with the two-wide operations as two correctly rounded ones.
#include <cmath>
#include <cstdint>

struct float2 {
  float x, y;
};
static inline float2 make_float2(float x, float y) { return {x, y}; }
static inline float2 __ffma2_rn(float2 a, float2 b, float2 c) { return {std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y)}; }
static inline float2 __fadd2_rn(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
static inline float2 __fmul2_rn(float2 a, float2 b) { return {a.x * b.x, a.y * b.y}; }
#define TENO_CERT_PAIRS
#include "teno_cert.cuh"

// v: n x 2 x 5 values, d: n x 2; out: n x 2 masks (the paired one, two single ones)
extern "C" void cert_pairs(int64_t n, const float* v, const float* d, float thr_f, float eps4_f, int* out) {
  for (int64_t i = 0; i < n; ++i) {
    const float* a = v + 10 * i;
    const float* b = a + 5;
    float2 p[5];
    for (int k = 0; k < 5; ++k) p[k] = {a[k], b[k]};
    out[2 * i] = int(teno_cert::certify_open2(p[0], p[1], p[2], p[3], p[4], {d[2 * i], d[2 * i + 1]}, thr_f, eps4_f));
    const bool ka = teno_cert::certify_keep(a[0], a[1], a[2], a[3], a[4], d[2 * i], thr_f, eps4_f);
    const bool kb = teno_cert::certify_keep(b[0], b[1], b[2], b[3], b[4], d[2 * i + 1], thr_f, eps4_f);
    out[2 * i + 1] = (ka ? 0 : 1) | (kb ? 0 : 2);
  }
}
