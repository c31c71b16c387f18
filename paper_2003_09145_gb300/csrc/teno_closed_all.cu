// teno_closed_all.cu -- the closed-form pass of every direction in one launch,
// for grids whose interfaces of one direction do not fill the chip, and the
// passes without binary32 planes for the largest grids (a translation unit of
// its own: it compiles in parallel with the per-direction kernels).
#include <cstdint>
#include <cuda_runtime.h>

#include "teno.h"
#include "teno_faces.cuh"
#include "teno_launch.h"

namespace teno {

// Every direction in one launch (blockIdx.y: the direction), each with its own
// fluxes, list and counter.  Measured (us per step, a launch per direction
// against one): 172 against 153 at 100 x 300, 344 against 298 at 32^3, 208
// against 202 at 129 x 515 with walls; 852 against 867 at 64^3, so the line is
// drawn at kClosedAllCells.
template <int NDIM, int WALL>
__global__ void __launch_bounds__(128, TENO_CLOSED_MINBLOCKS) flux_closed_all_kernel(
    const double* __restrict__ U, const double* __restrict__ aux, const double* __restrict__ fh,
    const float4* __restrict__ pf, const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat,
    int64_t fstride, uint2* __restrict__ list, int64_t lstride, unsigned* __restrict__ count,
    int* __restrict__ status, Grid G, Scheme S) {
  const int d = blockIdx.y;
  Fhat += d * fstride;
  list += d * lstride;
  count += d;
  if (d == 0) closed_faces<NDIM, 0, WALL, false>(U, aux, fh, pf, alpha_bits, Fhat, list, count, status, G, S, nullptr);
  if constexpr (NDIM > 1)
    if (d == 1) closed_faces<NDIM, 1, WALL, false>(U, aux, fh, pf, alpha_bits, Fhat, list, count, status, G, S, nullptr);
  if constexpr (NDIM > 2)
    if (d == 2) closed_faces<NDIM, 2, WALL, false>(U, aux, fh, pf, alpha_bits, Fhat, list, count, status, G, S, nullptr);
}

cudaError_t launch_closed_all(int ndim, const double* U, const double* aux, const double* fh, const float4* pf,
                              const unsigned long long* alpha, double* Fhat, int64_t fstride, uint2* list,
                              int64_t lstride, unsigned* count, int* status, const Grid& G, const Scheme& S, int nsm,
                              cudaStream_t st) {
  int64_t nifc = 0;
  bool plain = true;
  for (int d = 0; d < ndim; ++d) {
    int64_t m = 1;
    for (int k = 0; k < 3; ++k) m *= G.n[k] + (k == d ? 1 : 0);
    nifc = m > nifc ? m : nifc;
    plain = plain && G.bc[d] < TENO_BC_REFLECTIVE;
  }
  int64_t blocks = (nifc + 127) / 128;
  if (blocks > int64_t(nsm) * 64) blocks = int64_t(nsm) * 64;
  const dim3 grid{static_cast<unsigned>(blocks), static_cast<unsigned>(ndim), 1u};
  if (ndim == 2) {
    if (plain) flux_closed_all_kernel<2, 0><<<grid, 128, 0, st>>>(U, aux, fh, pf, alpha, Fhat, fstride, list, lstride, count, status, G, S);
    else flux_closed_all_kernel<2, 3><<<grid, 128, 0, st>>>(U, aux, fh, pf, alpha, Fhat, fstride, list, lstride, count, status, G, S);
  } else {
    if (plain) flux_closed_all_kernel<3, 0><<<grid, 128, 0, st>>>(U, aux, fh, pf, alpha, Fhat, fstride, list, lstride, count, status, G, S);
    else flux_closed_all_kernel<3, 3><<<grid, 128, 0, st>>>(U, aux, fh, pf, alpha, Fhat, fstride, list, lstride, count, status, G, S);
  }
  return cudaGetLastError();
}

// One direction on a grid of more than kPlaneCells cells, which keeps no planes
// and a list of indices: the conversions at each of the stencil's points, and
// every reconstruction of a listed interface decided -- the same fluxes.
template <int NDIM, int DIR, int WALL>
__global__ void __launch_bounds__(128, 3) flux_closed_noplanes_kernel(
    const double* __restrict__ U, const double* __restrict__ aux, const double* __restrict__ fh,
    const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat, uint32_t* __restrict__ list,
    unsigned* __restrict__ count, int* __restrict__ status, Grid G, Scheme S) {
  closed_faces<NDIM, DIR, WALL, false, false>(U, aux, fh, nullptr, alpha_bits, Fhat, list, count, status, G, S,
                                              nullptr);
}
template <int NDIM, int DIR, bool GH>
__global__ void __launch_bounds__(128) flux_correct_noplanes_kernel(
    const double* __restrict__ U, const double* __restrict__ aux,
    const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat, const uint32_t* __restrict__ list,
    const unsigned* __restrict__ count, int* __restrict__ status, Grid G, Scheme S, int nsm) {
  __shared__ CorrectScratch<NDIM> scratch[4];
  correct_list<NDIM, DIR, GH>(U, aux, alpha_bits, Fhat, list, *count, status, G, S, nsm, scratch[threadIdx.x >> 5]);
}

template <int NDIM, int DIR>
static void noplanes_dir(const double* U, const double* aux, const double* fh, const unsigned long long* alpha,
                         double* Fhat, uint32_t* list, unsigned* count, int* status, const Grid& G, const Scheme& S,
                         int nsm, int blocks, int cblocks, cudaStream_t st) {
  // (WALL 1 also covers plain boundaries: the mirror flags are then 0)
  if (G.bc[DIR] == TENO_BC_DIRICHLET) {
    flux_closed_noplanes_kernel<NDIM, DIR, 2><<<blocks, 128, 0, st>>>(U, aux, fh, alpha, Fhat, list, count, status, G, S);
    flux_correct_noplanes_kernel<NDIM, DIR, true><<<cblocks, 128, 0, st>>>(U, aux, alpha, Fhat, list, count, status, G, S, nsm);
  } else {
    flux_closed_noplanes_kernel<NDIM, DIR, 1><<<blocks, 128, 0, st>>>(U, aux, fh, alpha, Fhat, list, count, status, G, S);
    flux_correct_noplanes_kernel<NDIM, DIR, false><<<cblocks, 128, 0, st>>>(U, aux, alpha, Fhat, list, count, status, G, S, nsm);
  }
}

void launch_flux_noplanes(int ndim, int dir, const double* U, const double* aux, const double* fh,
                          const unsigned long long* alpha, double* Fhat, uint32_t* list, unsigned* count, int* status,
                          const Grid& G, const Scheme& S, int nsm, int blocks, int cblocks, cudaStream_t st) {
  auto* f = ndim == 1 ? noplanes_dir<1, 0>
            : ndim == 2 ? (dir == 0 ? noplanes_dir<2, 0> : noplanes_dir<2, 1>)
                        : (dir == 0 ? noplanes_dir<3, 0> : (dir == 1 ? noplanes_dir<3, 1> : noplanes_dir<3, 2>));
  f(U, aux, fh, alpha, Fhat, list, count, status, G, S, nsm, blocks, cblocks, st);
}

}  // namespace teno
