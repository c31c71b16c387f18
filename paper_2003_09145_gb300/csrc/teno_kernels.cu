// teno_kernels.cu -- sm_103a kernels of the TENO5-LAD Euler right-hand side
// and the SSP-RK3 stage updates (all FP64).
//
// One right-hand-side evaluation L(U) (eq. 2.2) is
//   cell_kernel    : per cell, primitive variables (u_k, p) and the Roe weights
//                    sqrt(rho), (E + p)/sqrt(rho); the global Lax-Friedrichs
//                    speeds alpha_{d,s} = max |lambda_s| of every direction
//                    (warp-shuffle max, block max, one atomic per block);
//   flux_closed_kernel<D>, flux_correct_kernel<D> : per interface of direction
//                    D the flux with every stencil kept and the certified test,
//                    then the differences that the open reconstructions' cut
//                    stencils make (flux_kernel<D>: both in one pass, with
//                    the selections' flags; flux_wenoz_kernel<D>: WENO-Z);
//   diff_kernel<D> : per cell, -(F^_{i+1/2} - F^_{i-1/2}) / dx_D, written,
//                    accumulated, or fused into the SSP-RK3 stage (eq. 4.1-4.3).
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

#include "teno_closed.cuh"
#include "teno_device.cuh"
#include "teno_faces.cuh"
#include "teno_flux.cuh"
#include "teno_launch.h"

namespace teno {

// ---------------------------------------------------------------------------
// Cell pass: primitive variables, Roe weights and LF speeds.
// The primitive variables come from one reciprocal square root per cell
// (cell_primitives); the wave speeds |u_d - c|, |u_d|, |u_d + c| are reduced
// to their maxima over all cells.
// aux layout: [aux_fields(ndim) = 2 ndim + 3][ncell]: u_0/2..u_{ndim-1}/2,
// p/2, sqrt(rho), (E+p)/sqrt(rho), m_0/sqrt(rho)..m_{ndim-1}/sqrt(rho).
// With `fh`, also the binary32 copies `pf` (store_planes) and the half physical fluxes F_d/2 (eq. 4.7)
// of every direction, momentum and energy components only (the mass one is
// m_d/2), [ndim][nvar - 1][ncell], for the closed-form flux pass.
// alpha layout (bit patterns of non-negative doubles): [ndim][3] =
// max|u_d - c|, max|u_d|, max|u_d + c|.
// ---------------------------------------------------------------------------
// F_d/2 of cell c for d = D..NDIM-1 into fh[d][v - 1][c], v = 1..nvar-1.
// The off-diagonal momentum fluxes rho u_d u_k are formed once, as (u_d/2) m_k
// of the lower d, for both directions.
template <int NDIM, int D>
__device__ __forceinline__ void store_flux_half(const double (&Uc)[NDIM + 2], const double (&uh)[NDIM], double pn,
                                                double ep, double* __restrict__ fh, int64_t ncell, int64_t c) {
  if constexpr (D < NDIM) {
    constexpr int NVAR = NDIM + 2;
    double Fh[NVAR];
    cell_flux_half_ep<NDIM, D>(Uc, uh[D], pn, ep, Fh);
#pragma unroll
    for (int k = 0; k < D; ++k) Fh[1 + k] = uh[k] * Uc[1 + D];
#pragma unroll
    for (int v = 1; v < NVAR; ++v) fh[(int64_t)(D * (NVAR - 1) + v - 1) * ncell + c] = Fh[v];
    store_flux_half<NDIM, D + 1>(Uc, uh, pn, ep, fh, ncell, c);
  }
}

#ifndef TENO_CELL_MINBLOCKS
#define TENO_CELL_MINBLOCKS 2   // 128 registers, 16 warps per SM: measured 0.1 ms per step
#endif                          // faster than 3 (80 registers) or 4 (64)
// With ARG, every block also writes, per speed, its largest value and the
// lowest cell index attaining it to cand[block][9][2] (value bits, index):
// the arg-max cells through which the adjoint differentiates the global
// speeds (argmax_finish_kernel reduces the candidates).
template <int NDIM, bool ARG>
__global__ void __launch_bounds__(256, TENO_CELL_MINBLOCKS) cell_kernel(const double* __restrict__ U,
                                                   double* __restrict__ aux,
                                                   double* __restrict__ fh, float4* __restrict__ pf,
                                                   unsigned long long* __restrict__ alpha,
                                                   int* __restrict__ status,
                                                   int64_t ncell, double gamma,
                                                   unsigned long long* __restrict__ cand) {
  constexpr int NVAR = NDIM + 2;
  unsigned long long lam[NDIM][3];   // bit patterns of the running maxima (>= 0)
  long long arg[NDIM][3];            // (ARG) the first cell of this thread attaining each
#pragma unroll
  for (int d = 0; d < NDIM; ++d)
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      lam[d][s] = 0ull;
      arg[d][s] = ncell;
    }
  bool bad = false;
  // the block's running maxima so far, as binary32 values not above them
  __shared__ volatile float low[NDIM * 3];
  if (threadIdx.x < NDIM * 3) low[threadIdx.x] = -1.0f;
  __syncthreads();
  const float gamma_f = static_cast<float>(gamma);
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    double uh[NDIM], p, hr, ep;
    if (!cell_primitives<NDIM>(U, ncell, c, gamma, aux, uh, ep, p, hr)) bad = true;
    if (fh) {
      double Uc[NVAR];
#pragma unroll
      for (int v = 0; v < NVAR; ++v) Uc[v] = U[v * ncell + c];
      const double pn = aux[NDIM * ncell + c];
      store_flux_half<NDIM, 0>(Uc, uh, pn, ep, fh, ncell, c);
    }
    if (pf) {
      double Uc[NVAR], su[NDIM];
#pragma unroll
      for (int v = 0; v < NVAR; ++v) Uc[v] = U[v * ncell + c];
#pragma unroll
      for (int k = 0; k < NDIM; ++k) su[k] = aux[(NDIM + 3 + k) * ncell + c];
      store_planes<NDIM>(pf, ncell, c, Uc, uh, aux[NDIM * ncell + c], aux[(NDIM + 1) * ncell + c],
                         aux[(NDIM + 2) * ncell + c], su);
    }
    // The wave speeds only enter through their maxima: a cell whose binary32
    // upper bounds all lie below the block's maxima is skipped (15 of a 3D
    // cell's FP64 instructions; with the halvings and doublings on the integer
    // pipe and the off-diagonal momentum fluxes formed once the pass fell from
    // 476 to 406 us at 160^3, FP64 pipe 82 % busy, and a 256^3 step from 24.3
    // to 22.5 ms).  Anything not certainly below -- NaN too -- is
    // evaluated, so the maxima are those of all cells, bit for bit.
    float ub[NDIM][3];
    speed_bounds<NDIM>(uh, p, hr, gamma_f, ub);
    bool below = true;
#pragma unroll
    for (int d = 0; d < NDIM; ++d)
#pragma unroll
      for (int s = 0; s < 3; ++s) below = below && ub[d][s] < low[d * 3 + s];
    if (below) continue;
    double cs;
    if (!sound_speed(p, hr, gamma, cs)) bad = true;
    // u -+ c = 2 (u/2) -+ c with one rounding, as a subtraction of u would;
    // max|u| is kept as max|u/2| and doubled (exactly) below
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
      const double x[3] = {fma(2.0, uh[d], -cs), uh[d], fma(2.0, uh[d], cs)};
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const unsigned long long m = max_abs_bits(lam[d][s], x[s]);
        if constexpr (ARG)
          if (m != lam[d][s]) arg[d][s] = c;
        if (m != lam[d][s]) {
          lam[d][s] = m;
          // (hi_float truncates, so the published value is not above the
          // maximum; a lost update only leaves a lower bound)
          const float f = (s == 1 ? 2.0f : 1.0f) * hi_float(__longlong_as_double(static_cast<long long>(m)));
          if (f > low[d * 3 + s] && f > 0x1p-100f && f < 0x1p100f) low[d * 3 + s] = f;
        }
      }
    }
  }
#pragma unroll
  for (int d = 0; d < NDIM; ++d) lam[d][1] = dbits(2.0 * __longlong_as_double(static_cast<long long>(lam[d][1])));
  // warp max on bit patterns (all values are >= 0); with ARG the lowest
  // index among the lanes holding the maximum
  __shared__ unsigned long long red[8][NDIM * 3];
  __shared__ long long rarg[ARG ? 8 : 1][NDIM * 3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int d = 0; d < NDIM; ++d)
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      unsigned long long v = lam[d][s];
      long long a = arg[d][s];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        if constexpr (ARG) {
          const long long b = __shfl_xor_sync(0xffffffffu, a, o);
          if (w > v || (w == v && b < a)) a = b;
        }
        v = v > w ? v : w;
      }
      if (lane == 0) {
        red[warp][d * 3 + s] = v;
        if constexpr (ARG) rarg[warp][d * 3 + s] = a;
      }
    }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, kStatusNonphysical);
  __syncthreads();
  if (threadIdx.x < NDIM * 3) {
    unsigned long long v = 0;
    long long a = ncell;
    const int nw = blockDim.x >> 5;
    for (int w = 0; w < nw; ++w) {
      const unsigned long long x = red[w][threadIdx.x];
      if constexpr (ARG) {
        const long long b = rarg[w][threadIdx.x];
        if (x > v || (x == v && b < a)) a = b;
      }
      v = v > x ? v : x;
    }
    atomicMax(&alpha[threadIdx.x], v);
    if constexpr (ARG) {
      cand[(blockIdx.x * 9 + threadIdx.x) * 2] = v;
      cand[(blockIdx.x * 9 + threadIdx.x) * 2 + 1] = static_cast<unsigned long long>(a);
    }
  }
}

// The arg-max cells of the nine LF speeds from the cell pass's per-block
// candidates: the largest value of each speed and the lowest cell index
// attaining it (entries of unused directions stay as they are).
// One warp per speed (one block-wide reduction after another took 16 us).
constexpr int kArgThreads = 288;
__global__ void __launch_bounds__(kArgThreads) argmax_finish_kernel(const unsigned long long* __restrict__ cand,
                                                                    int nblocks, int nspeed,
                                                                    unsigned long long* __restrict__ argidx) {
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  if (k >= nspeed) return;
  unsigned long long v = 0, a = ~0ull;
  for (int b = lane; b < nblocks; b += 32) {
    const unsigned long long x = cand[(b * 9 + k) * 2], i = cand[(b * 9 + k) * 2 + 1];
    if (x > v || (x == v && i < a)) {
      v = x;
      a = i;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_down_sync(0xffffffffu, v, o), i = __shfl_down_sync(0xffffffffu, a, o);
    if (x > v || (x == v && i < a)) {
      v = x;
      a = i;
    }
  }
  if (lane == 0) argidx[k] = a;
}

// ---------------------------------------------------------------------------
// Interface fluxes of direction DIR.
// ---------------------------------------------------------------------------

// What bounds it: FP64 issue.  Against the whole characteristic values at every
// interface (whose error on a 1e5 Pa state is 1.2e-13 of the flux scale, not 3e-14)
// the all-kept flux costs up to a tenth where many selections cut and nothing
// where few do: right-hand sides with flags at 160^3 12.7 against 12.8 ms, 1024^2
// 1.97 / 1.91, 64^3 1.20 / 1.09, 4096 cells 39 / 37 us; with the all-kept sums as
// chains of half fluxes formed here 14.1, 2.18, 1.21 ms, 40 us.
#ifndef TENO_FLUX_MINBLOCKS
#define TENO_FLUX_MINBLOCKS 4
#endif

template <int NDIM, int DIR, bool WITH_FLAGS, bool GH>
__global__ void __launch_bounds__(128, TENO_FLUX_MINBLOCKS) flux_kernel(
    const double* __restrict__ U, const double* __restrict__ aux, const double* __restrict__ fh,
    const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat,
    uint8_t* __restrict__ flags, int* __restrict__ status, Grid G, Scheme S) {
  constexpr int NVAR = NDIM + 2;
  // interface grid: n along the other axes, n_DIR + 1 along DIR
  const int64_t m0 = G.n[0] + (DIR == 0), m1 = G.n[1] + (DIR == 1), m2 = G.n[2] + (DIR == 2);
  const int64_t nifc = m0 * m1 * m2;
  const int64_t ncell = G.ncell;
  const int64_t stride_d = (DIR == 0) ? 1 : (DIR == 1 ? G.n[0] : G.n[0] * G.n[1]);
  const int64_t nd = G.n[DIR];
  const int bcd = G.bc[DIR];

  double alpha[NVAR];
  {
    double am = __longlong_as_double((long long)alpha_bits[DIR * 3 + 0]);
    double a0 = __longlong_as_double((long long)alpha_bits[DIR * 3 + 1]);
    double ap = __longlong_as_double((long long)alpha_bits[DIR * 3 + 2]);
    alpha[0] = 0.5 * am;
#pragma unroll
    for (int f = 1; f < NVAR - 1; ++f) alpha[f] = 0.5 * a0;
    alpha[NVAR - 1] = 0.5 * ap;
  }
  double nal[NVAR];
#pragma unroll
  for (int f = 0; f < NVAR; ++f) nal[f] = -2.0 * alpha[f];

  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nifc;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i0 = q % m0;
    const int64_t r = q / m0;
    const int64_t i1 = r % m1;
    const int64_t i2 = r / m1;
    const int64_t id = (DIR == 0) ? i0 : (DIR == 1 ? i1 : i2);
    // linear index of the cell with coordinate 0 along DIR on this line
    const int64_t base = (DIR == 0) ? (i2 * G.n[1] + i1) * G.n[0]
                       : (DIR == 1) ? i2 * G.n[1] * G.n[0] + i0
                                    : i1 * G.n[0] + i0;

    int64_t cells[6];
    unsigned flips = 0u;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      bool f;
      const int64_t k = id - 3 + j;
      cells[j] = (GH && (k < 0 || k >= nd)) ? ncell + 2 * DIR + (k >= nd) : base + ghost(k, nd, bcd, f) * stride_d;
      flips |= GH ? 0u : unsigned(f) << j;
    }
    double out[NVAR];
    unsigned fl[NVAR][2];
    interface_flux<NDIM, DIR, WITH_FLAGS, kFluxFull, GH>(U, aux, ncell, cells, flips, alpha, nal, S, out, fl, status,
                                                        GhostCells{G.gU, G.gaux, G.gfh, G.gpf}, fh);
    if (WITH_FLAGS) {
      // direction block offset is applied by the caller through `flags`
#pragma unroll
      for (int s = 0; s < NVAR; ++s)
#pragma unroll
        for (int side = 0; side < 2; ++side)
          flags[(int64_t)(s * 2 + side) * nifc + q] = (uint8_t)fl[s][side];
    }
#pragma unroll
    for (int v = 0; v < NVAR; ++v) Fhat[(int64_t)v * nifc + q] = out[v];
  }
}

template <int NDIM, int DIR, int WALL, bool ROE = false>
__global__ void __launch_bounds__(128, TENO_CLOSED_MINBLOCKS) flux_closed_kernel(
    const double* __restrict__ U, const double* __restrict__ aux, const double* __restrict__ fh,
    const float4* __restrict__ pf, const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat,
    uint2* __restrict__ list, unsigned* __restrict__ count, int* __restrict__ status, Grid G,
    Scheme S, double* __restrict__ roe_out = nullptr) {
  closed_faces<NDIM, DIR, WALL, ROE>(U, aux, fh, pf, alpha_bits, Fhat, list, count, status, G, S, roe_out);
}

template <int NDIM, int DIR, bool GH>
__global__ void __launch_bounds__(128) flux_correct_kernel(
    const double* __restrict__ U, const double* __restrict__ aux,
    const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat,
    const uint2* __restrict__ list, const unsigned* __restrict__ count, int* __restrict__ status,
    Grid G, Scheme S, int nsm) {
  __shared__ CorrectScratch<NDIM> scratch[4];
  correct_list<NDIM, DIR, GH>(U, aux, alpha_bits, Fhat, list, *count, status, G, S, nsm, scratch[threadIdx.x >> 5]);
}

// The lists of every direction in one launch (blockIdx.y: the direction), each
// with its own fluxes and list (stages of small and medium grids).
template <int NDIM, bool GH>
__global__ void __launch_bounds__(128) flux_correct_all_kernel(
    const double* __restrict__ U, const double* __restrict__ aux,
    const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat, int64_t fstride,
    const uint2* __restrict__ list, int64_t lstride, const unsigned* __restrict__ count, int* __restrict__ status,
    Grid G, Scheme S, int nsm) {
  __shared__ CorrectScratch<NDIM> scratch[4];
  CorrectScratch<NDIM>& W = scratch[threadIdx.x >> 5];
  const int d = blockIdx.y;
  const int64_t n = count[d];
  Fhat += d * fstride;
  list += d * lstride;
  if (d == 0) correct_list<NDIM, 0, GH>(U, aux, alpha_bits, Fhat, list, n, status, G, S, nsm, W);
  if constexpr (NDIM > 1)
    if (d == 1) correct_list<NDIM, 1, GH>(U, aux, alpha_bits, Fhat, list, n, status, G, S, nsm, W);
  if constexpr (NDIM > 2)
    if (d == 2) correct_list<NDIM, 2, GH>(U, aux, alpha_bits, Fhat, list, n, status, G, S, nsm, W);
}

template <int NDIM, int DIR, bool GH>
__global__ void __launch_bounds__(128) flux_wenoz_kernel(
    const double* __restrict__ U, const double* __restrict__ aux,
    const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat, int* __restrict__ status,
    Grid G, Scheme Sx) {
  constexpr int NVAR = NDIM + 2;
  Scheme S = Sx;
  S.variant = kSchemeWenoZ;   // known to the compiler: the cutoffs' code folds away
  S.keep_idx = -1;
  const int64_t nifc = (G.n[0] + (DIR == 0)) * (G.n[1] + (DIR == 1)) * (G.n[2] + (DIR == 2));
  double alpha[NVAR], nal[NVAR];
  half_speeds<NDIM, DIR>(alpha_bits, alpha, nal);
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nifc; q += (int64_t)gridDim.x * blockDim.x) {
    uint32_t cells[6];
    unsigned flips;
    interface_cells<NDIM, DIR, GH>(static_cast<uint32_t>(q), G, cells, flips);
    double out[NVAR];
    unsigned fl[NVAR][2];
    interface_flux<NDIM, DIR, false, kFluxChar, GH>(U, aux, G.ncell, cells, flips, alpha, nal, S, out, fl, status,
                                                   GhostCells{G.gU, G.gaux, G.gfh, G.gpf});
#pragma unroll
    for (int v = 0; v < NVAR; ++v) Fhat[(int64_t)v * nifc + q] = out[v];
  }
}

// ---------------------------------------------------------------------------
// Conservative difference (eq. 2.2) and SSP-RK3 stage update (eq. 4.1-4.3).
// With t_d = F^_{i-1/2} - F^_{i+1/2} of direction d and r_d = dx_0 / dx_d,
// L(U) = (t_0 + r_1 t_1 + r_2 t_2) / dx_0: R carries the unscaled partial
// sum and 1/dx_0 is applied once (in the stage's coefficient, or at the end
// of a plain right-hand side), one FP64 instruction fewer per element than
// scaling every direction -- the passes are bound by FP64 issue.  The
// fluxes arrive as kFluxScale F^ (teno_flux.cuh), so that factor is
// divided out with dx_0 (dx_0 below stands for kFluxScale dx_0).
// MODE (a template argument, so that every load of a cell is issued before
// its stores):
//   kDiffFirst  R = t_0                        (first of several directions)
//   kDiffAcc    R += r_d t_d                   (a middle direction)
//   kDiffRhs    R = (R + r_d t_d) / dx_0       (last direction of a plain RHS;
//                                               R = t_0 / dx_0 in 1D)
//   2, 3, 4     with s = R + r_d t_d (t_0 in 1D) and c = dt / dx_0:
//               2: U1 = Un + c s;  3: U2 = 3/4 Un + 1/4 U1 + 1/4 c s;
//               4: Un <- 1/3 Un + 2/3 U2 + 2/3 c s.
// ---------------------------------------------------------------------------
constexpr int kDiffFirst = 0, kDiffAcc = 1, kDiffRhs = 5;

// GRAV (last direction only): the body-force source of Sec. 4.3.2,
// S = (0, rho g, rho u.g), is added from the stage input Usrc.
template <int NDIM, int DIR, int MODE, bool GRAV = false>
__global__ void __launch_bounds__(256) diff_kernel(
    const double* __restrict__ Fhat, double* __restrict__ R,
    const double* Un, const double* Uk,   // not restrict: stage 3 writes Uout = Un in place
    double* Uout, const double* __restrict__ dt_ptr, Grid G, const double* Usrc) {
  constexpr bool stage = MODE >= 2 && MODE <= 4;
  constexpr bool acc = DIR > 0;   // R holds the earlier directions' sum
  constexpr int NVAR = NDIM + 2;
  const int64_t ncell = G.ncell;
  const int64_t m0 = G.n[0] + (DIR == 0), m1 = G.n[1] + (DIR == 1);
  const int64_t nifc = m0 * m1 * (G.n[2] + (DIR == 2));
  const double rd = G.rdx[DIR];
  // the interface fluxes are stored as kFluxScale F^: the last direction
  // divides by it together with dx_0
  const double idf = G.inv_dx[0] / kFluxScale;
  double c = 0.0;
  if (stage) {
    const double dt = *dt_ptr;
    if (!(dt > 0.0)) {
      // t >= t_end: the state is left unchanged.  The stage buffers U1, U2
      // take U^n, so that the stages after this one read defined values.
      if (MODE <= 3)
        for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < NVAR * ncell;
             e += (int64_t)gridDim.x * blockDim.x)
          Uout[e] = Un[e];
      return;
    }
    c = dt * idf;
  }
  // The interface left of cell c = (i2 n1 + i1) n0 + i0 is (i2 m1 + i1) m0 + i0:
  // x: c plus the row index c / n0 (one more interface per row); y: c plus
  // n0 times the plane index c / (n0 n1); z: c itself.
  const int64_t span = DIR == 0 ? G.n[0] : G.n[0] * G.n[1];
  const int64_t shift = DIR == 0 ? 1 : G.n[0];
  const bool narrow = ncell <= int64_t(UINT32_MAX);   // 32-bit division suffices
  for (int64_t cc = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; cc < ncell;
       cc += (int64_t)gridDim.x * blockDim.x) {
    int64_t left = cc;
    if (DIR < 2) {
      const int64_t q = narrow ? int64_t(uint32_t(cc) / uint32_t(span)) : cc / span;
      left += q * shift;
    }
    const int64_t right = left + (DIR == 0 ? 1 : (DIR == 1 ? m0 : m0 * m1));
    // all loads of the cell first
    double s[NVAR];
#pragma unroll
    for (int v = 0; v < NVAR; ++v) s[v] = Fhat[v * nifc + left] - Fhat[v * nifc + right];
    if (acc)
#pragma unroll
      for (int v = 0; v < NVAR; ++v) s[v] = fma(rd, s[v], R[v * ncell + cc]);
    double src[NVAR];
    if (GRAV) {
      const double rho = Usrc[cc];
      double w = 0.0;
      src[0] = 0.0;
#pragma unroll
      for (int k = 0; k < NDIM; ++k) {
        src[1 + k] = rho * G.grav[k];
        w = fma(Usrc[(1 + k) * ncell + cc], G.grav[k], w);
      }
      src[NVAR - 1] = w;
      // L = s / (30 dx_0) + S: a stage takes c (s + 30 dx_0 S) with c = dt / (30 dx_0)
      if (stage)
#pragma unroll
        for (int v = 1; v < NVAR; ++v) s[v] = fma(kFluxScale * G.dx[0], src[v], s[v]);
    }
    if (MODE == kDiffFirst || MODE == kDiffAcc) {
#pragma unroll
      for (int v = 0; v < NVAR; ++v) R[v * ncell + cc] = s[v];
    } else if (MODE == kDiffRhs) {
#pragma unroll
      for (int v = 0; v < NVAR; ++v) R[v * ncell + cc] = GRAV ? fma(s[v], idf, src[v]) : s[v] * idf;
    } else {
      double o[NVAR];
#pragma unroll
      for (int v = 0; v < NVAR; ++v) o[v] = stage_value(MODE, c, s[v], Un, Uk, v * ncell + cc);
#pragma unroll
      for (int v = 0; v < NVAR; ++v) Uout[v * ncell + cc] = o[v];
    }
  }
}

// The differences of every direction and the last one's MODE in one pass
// (kDiffRhs or a stage 2, 3, 4), from one flux buffer per direction: the
// per-direction passes' operations in their order, with the partial sum in a
// register instead of R -- the same results bit for bit in one launch
// instead of ndim.
template <int NDIM, int DIR>
__device__ __forceinline__ void add_direction(const double* __restrict__ Fhat, int64_t fstride, const Grid& G,
                                              uint32_t c, double (&s)[NDIM + 2]) {
  if constexpr (DIR < NDIM) {
    const uint32_t n0 = static_cast<uint32_t>(G.n[0]), n01 = n0 * static_cast<uint32_t>(G.n[1]);
    const int64_t m0 = G.n[0] + (DIR == 0), m1 = G.n[1] + (DIR == 1);
    const int64_t nifc = m0 * m1 * (G.n[2] + (DIR == 2));
    const int64_t left = DIR == 0 ? (int64_t)c + c / n0 : (DIR == 1 ? (int64_t)c + (int64_t)(c / n01) * n0 : (int64_t)c);
    const int64_t right = left + (DIR == 0 ? 1 : (DIR == 1 ? m0 : m0 * m1));
    const double* F = Fhat + DIR * fstride;
#pragma unroll
    for (int v = 0; v < NDIM + 2; ++v) {
      const double t = F[v * nifc + left] - F[v * nifc + right];
      s[v] = DIR == 0 ? t : fma(G.rdx[DIR], t, s[v]);
    }
    add_direction<NDIM, DIR + 1>(Fhat, fstride, G, c, s);
  }
}

template <int NDIM, int MODE, bool GRAV>
__global__ void __launch_bounds__(256) diff_all_kernel(const double* __restrict__ Fhat, int64_t fstride,
                                                       double* R, const double* Un, const double* Uk, double* Uout,
                                                       const double* __restrict__ dt_ptr, Grid G,
                                                       const double* Usrc) {
  constexpr bool stage = MODE != kDiffRhs;
  constexpr int NVAR = NDIM + 2;
  const int64_t ncell = G.ncell;
  const double idf = G.inv_dx[0] / kFluxScale;
  double c = 0.0;
  if (stage) {
    const double dt = *dt_ptr;
    if (!(dt > 0.0)) {   // as diff_kernel
      if (MODE <= 3)
        for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < NVAR * ncell;
             e += (int64_t)gridDim.x * blockDim.x)
          Uout[e] = Un[e];
      return;
    }
    c = dt * idf;
  }
  for (int64_t cc = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; cc < ncell;
       cc += (int64_t)gridDim.x * blockDim.x) {
    double s[NVAR], src[NVAR];
    add_direction<NDIM, 0>(Fhat, fstride, G, static_cast<uint32_t>(cc), s);
    if (GRAV) {
      const double rho = Usrc[cc];
      double w = 0.0;
      src[0] = 0.0;
#pragma unroll
      for (int k = 0; k < NDIM; ++k) {
        src[1 + k] = rho * G.grav[k];
        w = fma(Usrc[(1 + k) * ncell + cc], G.grav[k], w);
      }
      src[NVAR - 1] = w;
      if (stage)
#pragma unroll
        for (int v = 1; v < NVAR; ++v) s[v] = fma(kFluxScale * G.dx[0], src[v], s[v]);
    }
    double o[NVAR];
#pragma unroll
    for (int v = 0; v < NVAR; ++v)
      o[v] = stage ? stage_value(MODE, c, s[v], Un, Uk, v * ncell + cc) : (GRAV ? fma(s[v], idf, src[v]) : s[v] * idf);
    double* out = stage ? Uout : R;
#pragma unroll
    for (int v = 0; v < NVAR; ++v) out[v * ncell + cc] = o[v];
  }
}

// ---------------------------------------------------------------------------
// Time step (eq. dt1 / dt2; harmonic 3D form) from the LF speeds of U^n:
// max_i(|u_d| + c) = max(max|u_d - c|, max|u_d + c|).  Clipped to t_end - t.
// ---------------------------------------------------------------------------
template <int NDIM>
__global__ void dt_kernel(const unsigned long long* __restrict__ alpha_bits,
                          Grid G, double cfl, double dt_fixed, double* t_dev,
                          double t_end, double* dt_ws, double* dt_out) {
  const double* dx = G.dx;
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double smax[3];
#pragma unroll
  for (int d = 0; d < NDIM; ++d) {
    unsigned long long a = alpha_bits[d * 3 + 0], b = alpha_bits[d * 3 + 2];
    smax[d] = __longlong_as_double((long long)(a > b ? a : b));
  }
  double dt;
  if (dt_fixed > 0.0) {
    dt = dt_fixed;
  } else if (NDIM == 1) {
    dt = cfl * dx[0] / smax[0];
  } else if (NDIM == 2) {
    const double dtx = dx[0] / smax[0], dty = dx[1] / smax[1];
    dt = cfl * dtx * dty / (dtx + dty);
  } else {
    double acc = 0.0;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) acc += smax[d] / dx[d];
    dt = cfl / acc;
  }
  const double t = *t_dev;
  const double rem = t_end - t;
  if (rem < dt) dt = rem;
  if (!(dt > 0.0)) dt = 0.0;
  *dt_ws = dt;
  if (dt_out) *dt_out = dt;
  *t_dev = t + dt;
}

// ---------------------------------------------------------------------------
// Scheme constants (host side)
// ---------------------------------------------------------------------------
Scheme make_scheme(double gamma, double H, double eps, int b_l, int b_u, int variant, int ct_m) {
  static const double kPow10Neg[16] = {1e-0, 1e-1, 1e-2,  1e-3,  1e-4,  1e-5,  1e-6,  1e-7,
                                       1e-8, 1e-9, 1e-10, 1e-11, 1e-12, 1e-13, 1e-14, 1e-15};
  Scheme S;
  std::memset(&S, 0, sizeof(S));
  S.variant = variant;
  S.m_fixed = ct_m;
  S.eps_a = kTeno5ACr * 0.9 / (1.0 - 0.9 * kTeno5ACr) * kTeno5AXi * kTeno5AXi;
  S.gamma = gamma;
  S.gm1 = gamma - 1.0;
  S.gm1_h = static_cast<float>(S.gm1);
  S.gm1_l = static_cast<float>(S.gm1 - static_cast<double>(S.gm1_h));
  S.eps = eps;
  S.eps4 = 4.0 * eps;
  S.b_l = b_l;
  S.b_u = b_u;
  S.keep_all = 0;
  S.keep_idx = -1;
  if (variant == kSchemeLad) {
    const int K = b_u - b_l;
    S.nthr = K;
    S.top = 1;
    while (S.top * 2 <= K) S.top *= 2;
    // floor(theta K) >= j  <=>  max chi~ <= H (K/j - 1)   (eq. 3.1-3.2)
    for (int j = 1; j < K; ++j) S.thr[j - 1] = H * (double(K) / double(j) - 1.0);
    // theta == 1 in binary64  <=>  max chi~ / H <= 2^-53
    S.thr[K - 1] = H * 0x1p-53;
    // All stencils are kept whenever 3 (1 + max chi~)^6 C_T < 1 (then
    // chi_k >= gamma_min / (3 gamma_max) >= 1 / (3 (1 + max chi~)^6) > C_T); at
    // a given m, max chi~ <= thr[m - B_l - 1].  A relative margin of 1e-9 covers
    // the rounding of the threshold products.
    for (int c = 1; c <= K; ++c) {
      const int m = b_l + c;
      const double x = 1.0 + S.thr[c - 1];
      const double x6 = x * x * x * x * x * x;
      if (3.0 * x6 * kPow10Neg[m] <= 1.0 - 1e-9) S.keep_all |= 1u << m;
    }
    // the keep-all set is a suffix of B_l..B_u (the bound loosens as m grows)
    for (int c = 1; c <= K; ++c) {
      const unsigned suffix = ((1u << (b_u + 1)) - 1u) & ~((1u << (b_l + c)) - 1u);
      if (S.keep_all == suffix) {
        S.keep_idx = c - 1;
        break;
      }
    }
  } else if (variant == kSchemeTeno5 || variant == kSchemeTeno5A) {
    // The same bound with the largest C_T the scheme can take (TENO5: the
    // fixed one; TENO5-A: 1e-7): every stencil is kept when max chi~ <= thr
    // with 3 (1 + thr)^6 C_T <= 1 - 1e-9.
    const double ct = kPow10Neg[variant == kSchemeTeno5 ? ct_m : 7];
    double thr = std::pow(1.0 / (3.0 * ct), 1.0 / 6.0) - 1.0;
    for (int it = 0; it < 200 && thr > 0.0; ++it) {
      const double x = 1.0 + thr;
      if (3.0 * (x * x * x * x * x * x) * ct <= 1.0 - 1e-9) break;
      thr *= 1.0 - 1e-7;
    }
    if (thr > 0.0) {
      S.thr[0] = thr;
      S.keep_idx = 0;
    }
  }
  // (WENO-Z has no cutoff and no keep-all shortcut: keep_idx stays -1)
  for (int j = 0; j < kMaxLadder; ++j) S.thr_f[j] = static_cast<float>(S.thr[j]);
  // binary32 constants of the pre-test, rounded towards zero (conservative)
  auto down = [](double x) {
    float f = static_cast<float>(x);
    while (static_cast<double>(f) > x) f = std::nextafter(f, 0.0f);
    return std::nextafter(f, 0.0f);
  };
  // (the FP32 test's rounding analysis wants eps well inside the normal range;
  // thr_keep_f = 0 passes only all-zero stencils, which are kept exactly)
  S.eps4_f = down(4.0 * eps);
  S.thr_keep_f = (S.keep_idx >= 0 && 4.0 * eps >= 0x1p-100) ? down(S.thr[S.keep_idx]) : 0.0f;
  return S;
}

// ---------------------------------------------------------------------------
// Fixed-state ghost cells: one thread per face slot, the cell pass's formulas
// on the face states (kGhostSlots entries per field).
// ---------------------------------------------------------------------------
template <int NDIM>
__global__ void ghost_cell_kernel(GhostStates gs, unsigned mask, double* __restrict__ gU,
                                  double* __restrict__ gaux, double* __restrict__ gfh, float4* __restrict__ gpf,
                                  double gamma, int* __restrict__ status) {
  constexpr int NVAR = NDIM + 2;
  const int slot = threadIdx.x;
  if (slot >= kGhostSlots || !((mask >> slot) & 1u)) return;
  double Uc[NVAR];
#pragma unroll
  for (int v = 0; v < NVAR; ++v) gU[v * kGhostSlots + slot] = Uc[v] = gs.U[slot][v];
  double uh[NDIM], ep, p, hr, cs;
  const bool ok = cell_primitives<NDIM>(gU, kGhostSlots, slot, gamma, gaux, uh, ep, p, hr);
  if (!(sound_speed(p, hr, gamma, cs) && ok) && status) atomicOr(status, kStatusNonphysical);
  store_flux_half<NDIM, 0>(Uc, uh, gaux[NDIM * kGhostSlots + slot], ep, gfh, kGhostSlots, slot);
  double su[NDIM];
#pragma unroll
  for (int k = 0; k < NDIM; ++k) su[k] = gaux[(NDIM + 3 + k) * kGhostSlots + slot];
  store_planes<NDIM>(gpf, kGhostSlots, slot, Uc, uh, gaux[NDIM * kGhostSlots + slot],
                     gaux[(NDIM + 1) * kGhostSlots + slot], gaux[(NDIM + 2) * kGhostSlots + slot], su);
}

cudaError_t launch_ghost_cells(int ndim, const GhostStates& gs, unsigned mask, const Grid& G, double gamma,
                               cudaStream_t st) {
  double* gU = const_cast<double*>(G.gU);
  double* gaux = const_cast<double*>(G.gaux);
  double* gfh = const_cast<double*>(G.gfh);
  float4* gpf = const_cast<float4*>(G.gpf);
  switch (ndim) {
    case 1: ghost_cell_kernel<1><<<1, 32, 0, st>>>(gs, mask, gU, gaux, gfh, gpf, gamma, nullptr); break;
    case 2: ghost_cell_kernel<2><<<1, 32, 0, st>>>(gs, mask, gU, gaux, gfh, gpf, gamma, nullptr); break;
    default: ghost_cell_kernel<3><<<1, 32, 0, st>>>(gs, mask, gU, gaux, gfh, gpf, gamma, nullptr); break;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static inline int blocks_for(int64_t n, int threads, int cap) {
  int64_t b = (n + threads - 1) / threads;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return static_cast<int>(b);
}

// The cell pass's grid: the blocks that are resident at once, so that a block
// sees many cells and its running maxima settle (2 per SM against 8: 22.49
// against 22.62 ms per 256^3 step, 3.70 against 3.77 at 2048^2).
int cell_blocks(int64_t ncell, int nsm) { return blocks_for(ncell, 256, nsm * TENO_CELL_MINBLOCKS); }

cudaError_t launch_cell(int ndim, const double* U, double* aux, double* fh, float4* pf,
                        unsigned long long* alpha, int* status, int64_t ncell,
                        double gamma, int nsm, cudaStream_t st, unsigned long long* cand) {
  const int threads = 256;
  const int blocks = cell_blocks(ncell, nsm);
  if (cand) {
    switch (ndim) {
      case 1: cell_kernel<1, true><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, status, ncell, gamma, cand); break;
      case 2: cell_kernel<2, true><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, status, ncell, gamma, cand); break;
      default: cell_kernel<3, true><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, status, ncell, gamma, cand); break;
    }
    return cudaGetLastError();
  }
  switch (ndim) {
    case 1: cell_kernel<1, false><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, status, ncell, gamma, nullptr); break;
    case 2: cell_kernel<2, false><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, status, ncell, gamma, nullptr); break;
    default: cell_kernel<3, false><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, status, ncell, gamma, nullptr); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_argmax_finish(int ndim, const unsigned long long* cand, int64_t ncell, int nsm,
                                 unsigned long long* argidx, cudaStream_t st) {
  argmax_finish_kernel<<<1, kArgThreads, 0, st>>>(cand, cell_blocks(ncell, nsm), 3 * ndim, argidx);
  return cudaGetLastError();
}

template <int NDIM, int DIR>
static int flux_launch(int blocks, int threads, int pblocks, int nsm, cudaStream_t st, const double* U,
                       const double* aux, const double* fh, const float4* pf, const unsigned long long* alpha,
                       double* Fhat, uint8_t* flags, uint2* list, unsigned* count, int* status, const Grid& G,
                       const Scheme& S, double* roe_out, bool correct) {
  const bool gh = G.bc[DIR] == TENO_BC_DIRICHLET;
  if (flags || !list) {
    if (flags && gh) flux_kernel<NDIM, DIR, true, true><<<blocks, threads, 0, st>>>(U, aux, fh, alpha, Fhat, flags, status, G, S);
    else if (flags) flux_kernel<NDIM, DIR, true, false><<<blocks, threads, 0, st>>>(U, aux, fh, alpha, Fhat, flags, status, G, S);
    else if (gh) flux_kernel<NDIM, DIR, false, true><<<blocks, threads, 0, st>>>(U, aux, fh, alpha, Fhat, flags, status, G, S);
    else flux_kernel<NDIM, DIR, false, false><<<blocks, threads, 0, st>>>(U, aux, fh, alpha, Fhat, flags, status, G, S);
    return 1;
  }
  if (S.variant == kSchemeWenoZ) {
    if (gh) flux_wenoz_kernel<NDIM, DIR, true><<<pblocks, threads, 0, st>>>(U, aux, alpha, Fhat, status, G, S);
    else flux_wenoz_kernel<NDIM, DIR, false><<<pblocks, threads, 0, st>>>(U, aux, alpha, Fhat, status, G, S);
    return 1;
  }
  if (!pf) {
    launch_flux_noplanes(NDIM, DIR, U, aux, fh, alpha, Fhat, reinterpret_cast<uint32_t*>(list), count, status, G, S,
                         nsm, blocks, pblocks, st);
    return 2;
  }
  if (G.bc[DIR] == TENO_BC_REFLECTIVE)
    flux_closed_kernel<NDIM, DIR, 1><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, Fhat, list, count, status, G, S);
  else if (gh)
    flux_closed_kernel<NDIM, DIR, 2><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, Fhat, list, count, status, G, S);
  else if (roe_out)
    flux_closed_kernel<NDIM, DIR, 0, true><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, Fhat, list, count, status,
                                                                      G, S, roe_out);
  else
    flux_closed_kernel<NDIM, DIR, 0><<<blocks, threads, 0, st>>>(U, aux, fh, pf, alpha, Fhat, list, count, status, G, S);
  if (!correct) return 1;
  if (gh)
    flux_correct_kernel<NDIM, DIR, true><<<pblocks, threads, 0, st>>>(U, aux, alpha, Fhat, list, count, status, G, S, nsm);
  else
    flux_correct_kernel<NDIM, DIR, false><<<pblocks, threads, 0, st>>>(U, aux, alpha, Fhat, list, count, status, G, S, nsm);
  return 2;
}

cudaError_t launch_flux(int ndim, int dir, const double* U, const double* aux, const double* fh, const float4* pf,
                        const unsigned long long* alpha, double* Fhat,
                        uint8_t* flags, uint2* list, unsigned* count, int* status,
                        const Grid& G, const Scheme& S, int nsm, cudaStream_t st,
                        int* launches, double* roe_out, bool correct) {
  int64_t nifc = 1;
  for (int k = 0; k < 3; ++k) nifc *= G.n[k] + (k == dir ? 1 : 0);
  if (nifc > int64_t(UINT32_MAX)) list = nullptr;   // list entries are 32-bit
  if (!count || !fh) list = nullptr;
  const int threads = 128;
  const int blocks = blocks_for(nifc, threads, nsm * 64);
  const int pblocks = blocks_for(nifc, threads, nsm * 16);
  int n = 0;
  if (ndim == 1) n = flux_launch<1, 0>(blocks, threads, pblocks, nsm, st, U, aux, fh, pf, alpha, Fhat, flags, list, count, status, G, S, roe_out, correct);
  else if (ndim == 2) {
    if (dir == 0) n = flux_launch<2, 0>(blocks, threads, pblocks, nsm, st, U, aux, fh, pf, alpha, Fhat, flags, list, count, status, G, S, roe_out, correct);
    else n = flux_launch<2, 1>(blocks, threads, pblocks, nsm, st, U, aux, fh, pf, alpha, Fhat, flags, list, count, status, G, S, roe_out, correct);
  } else {
    if (dir == 0) n = flux_launch<3, 0>(blocks, threads, pblocks, nsm, st, U, aux, fh, pf, alpha, Fhat, flags, list, count, status, G, S, roe_out, correct);
    else if (dir == 1) n = flux_launch<3, 1>(blocks, threads, pblocks, nsm, st, U, aux, fh, pf, alpha, Fhat, flags, list, count, status, G, S, roe_out, correct);
    else n = flux_launch<3, 2>(blocks, threads, pblocks, nsm, st, U, aux, fh, pf, alpha, Fhat, flags, list, count, status, G, S, roe_out, correct);
  }
  if (launches) *launches = n;
  return cudaGetLastError();
}

cudaError_t launch_correct_all(int ndim, const double* U, const double* aux, const unsigned long long* alpha,
                               double* Fhat, int64_t fstride, const uint2* list, int64_t lstride,
                               const unsigned* count, int* status, const Grid& G, const Scheme& S, int nsm,
                               cudaStream_t st) {
  int64_t nifc = 0;
  bool gh = false;
  for (int d = 0; d < ndim; ++d) {
    int64_t m = 1;
    for (int k = 0; k < 3; ++k) m *= G.n[k] + (k == d ? 1 : 0);
    nifc = m > nifc ? m : nifc;
    gh = gh || G.bc[d] == TENO_BC_DIRICHLET;
  }
  const dim3 grid(unsigned(blocks_for(nifc, 128, nsm * 16)), unsigned(ndim));
  if (ndim == 2) {
    if (gh) flux_correct_all_kernel<2, true><<<grid, 128, 0, st>>>(U, aux, alpha, Fhat, fstride, list, lstride, count, status, G, S, nsm);
    else flux_correct_all_kernel<2, false><<<grid, 128, 0, st>>>(U, aux, alpha, Fhat, fstride, list, lstride, count, status, G, S, nsm);
  } else {
    if (gh) flux_correct_all_kernel<3, true><<<grid, 128, 0, st>>>(U, aux, alpha, Fhat, fstride, list, lstride, count, status, G, S, nsm);
    else flux_correct_all_kernel<3, false><<<grid, 128, 0, st>>>(U, aux, alpha, Fhat, fstride, list, lstride, count, status, G, S, nsm);
  }
  return cudaGetLastError();
}

template <int NDIM, bool GRAV>
static void diff_all_launch(int blocks, cudaStream_t st, const double* Fhat, int64_t fstride, double* R,
                            const double* Un, const double* Uk, double* Uout, const double* dt, const Grid& G, int mode,
                            const double* Usrc) {
  switch (mode) {
    case 0: diff_all_kernel<NDIM, kDiffRhs, GRAV><<<blocks, 256, 0, st>>>(Fhat, fstride, R, Un, Uk, Uout, dt, G, Usrc); break;
    case 2: diff_all_kernel<NDIM, 2, GRAV><<<blocks, 256, 0, st>>>(Fhat, fstride, R, Un, Uk, Uout, dt, G, Usrc); break;
    case 3: diff_all_kernel<NDIM, 3, GRAV><<<blocks, 256, 0, st>>>(Fhat, fstride, R, Un, Uk, Uout, dt, G, Usrc); break;
    default: diff_all_kernel<NDIM, 4, GRAV><<<blocks, 256, 0, st>>>(Fhat, fstride, R, Un, Uk, Uout, dt, G, Usrc); break;
  }
}

cudaError_t launch_diff_all(int ndim, const double* Fhat, int64_t fstride, double* R, const double* Un,
                            const double* Uk, double* Uout, const double* dt, const Grid& G, int mode, int nsm,
                            cudaStream_t st, const double* Usrc) {
  if (mode != 0 && (mode < 2 || mode > 4)) return cudaErrorInvalidValue;
  const int blocks = blocks_for(G.ncell, 256, nsm * 16);
  const bool g = G.has_grav;
  if (ndim == 2) (g ? diff_all_launch<2, true> : diff_all_launch<2, false>)(blocks, st, Fhat, fstride, R, Un, Uk, Uout, dt, G, mode, Usrc);
  else (g ? diff_all_launch<3, true> : diff_all_launch<3, false>)(blocks, st, Fhat, fstride, R, Un, Uk, Uout, dt, G, mode, Usrc);
  return cudaGetLastError();
}

template <int NDIM, int DIR, bool GRAV>
static void diff_launch_last(int blocks, int threads, cudaStream_t st, const double* Fhat, double* R,
                             const double* Un, const double* Uk, double* Uout, const double* dt, const Grid& G,
                             int mode, const double* Usrc) {
  switch (mode) {
    case 0: diff_kernel<NDIM, DIR, kDiffRhs, GRAV><<<blocks, threads, 0, st>>>(Fhat, R, Un, Uk, Uout, dt, G, Usrc); break;
    case 2: diff_kernel<NDIM, DIR, 2, GRAV><<<blocks, threads, 0, st>>>(Fhat, R, Un, Uk, Uout, dt, G, Usrc); break;
    case 3: diff_kernel<NDIM, DIR, 3, GRAV><<<blocks, threads, 0, st>>>(Fhat, R, Un, Uk, Uout, dt, G, Usrc); break;
    default: diff_kernel<NDIM, DIR, 4, GRAV><<<blocks, threads, 0, st>>>(Fhat, R, Un, Uk, Uout, dt, G, Usrc); break;
  }
}

template <int NDIM, int DIR>
static void diff_launch(int blocks, int threads, cudaStream_t st, const double* Fhat,
                        double* R, const double* Un, const double* Uk, double* Uout,
                        const double* dt, const Grid& G, int mode, const double* Usrc) {
  // the first of several directions starts R; a middle one adds to it
  if (DIR < NDIM - 1) {
    if (DIR == 0) diff_kernel<NDIM, DIR, kDiffFirst><<<blocks, threads, 0, st>>>(Fhat, R, Un, Uk, Uout, dt, G, Usrc);
    else diff_kernel<NDIM, DIR, kDiffAcc><<<blocks, threads, 0, st>>>(Fhat, R, Un, Uk, Uout, dt, G, Usrc);
    return;
  }
  if (G.has_grav) diff_launch_last<NDIM, DIR, true>(blocks, threads, st, Fhat, R, Un, Uk, Uout, dt, G, mode, Usrc);
  else diff_launch_last<NDIM, DIR, false>(blocks, threads, st, Fhat, R, Un, Uk, Uout, dt, G, mode, Usrc);
}

cudaError_t launch_diff(int ndim, int dir, const double* Fhat, double* R,
                        const double* Un, const double* Uk, double* Uout,
                        const double* dt, const Grid& G, int mode,
                        int nsm, cudaStream_t st, const double* Usrc) {
  if (mode != 0 && (mode < 2 || mode > 4)) return cudaErrorInvalidValue;
  const int threads = 256;
  const int blocks = blocks_for(G.ncell, threads, nsm * 16);
  if (ndim == 1) diff_launch<1, 0>(blocks, threads, st, Fhat, R, Un, Uk, Uout, dt, G, mode, Usrc);
  else if (ndim == 2) {
    if (dir == 0) diff_launch<2, 0>(blocks, threads, st, Fhat, R, Un, Uk, Uout, dt, G, mode, Usrc);
    else diff_launch<2, 1>(blocks, threads, st, Fhat, R, Un, Uk, Uout, dt, G, mode, Usrc);
  } else {
    if (dir == 0) diff_launch<3, 0>(blocks, threads, st, Fhat, R, Un, Uk, Uout, dt, G, mode, Usrc);
    else if (dir == 1) diff_launch<3, 1>(blocks, threads, st, Fhat, R, Un, Uk, Uout, dt, G, mode, Usrc);
    else diff_launch<3, 2>(blocks, threads, st, Fhat, R, Un, Uk, Uout, dt, G, mode, Usrc);
  }
  return cudaGetLastError();
}

cudaError_t launch_dt(int ndim, const unsigned long long* alpha, const Grid& G,
                      double cfl, double dt_fixed, double* t_dev, double t_end,
                      double* dt_ws, double* dt_out, cudaStream_t st) {
  switch (ndim) {
    case 1: dt_kernel<1><<<1, 32, 0, st>>>(alpha, G, cfl, dt_fixed, t_dev, t_end, dt_ws, dt_out); break;
    case 2: dt_kernel<2><<<1, 32, 0, st>>>(alpha, G, cfl, dt_fixed, t_dev, t_end, dt_ws, dt_out); break;
    default: dt_kernel<3><<<1, 32, 0, st>>>(alpha, G, cfl, dt_fixed, t_dev, t_end, dt_ws, dt_out); break;
  }
  return cudaGetLastError();
}

teno_status forward_stage(const teno_grid* g, char* ws, size_t status_off, size_t dt_off,
                          size_t alpha_off, size_t aux_off, size_t fh_off, size_t pf_off, size_t fhat_off,
                          size_t list_off, const double* U, double* R, int mode, const double* Un, const double* Uk,
                          double* Uout, cudaStream_t st, unsigned long long* cand, double* roe_out,
                          size_t roe_stride) {
  Grid G;
  for (int k = 0; k < 3; ++k) {
    G.n[k] = g->n[k];
    G.bc[k] = k < g->ndim ? g->bc[k] : 0;
    G.dx[k] = k < g->ndim ? g->dx[k] : 1.0;
    G.inv_dx[k] = 1.0 / G.dx[k];
    G.rdx[k] = G.dx[0] / G.dx[k];
  }
  G.ncell = g->n[0] * g->n[1] * g->n[2];
  const Scheme S = scheme_of(g);
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0)
    nsm = 152;
  int* status = reinterpret_cast<int*>(ws + status_off);
  const double* dt = reinterpret_cast<const double*>(ws + dt_off);
  auto* alpha = reinterpret_cast<unsigned long long*>(ws + alpha_off);
  double* aux = reinterpret_cast<double*>(ws + aux_off);
  double* Fhat = reinterpret_cast<double*>(ws + fhat_off);
  uint2* list = list_off ? reinterpret_cast<uint2*>(ws + list_off) : nullptr;
  double* fh = fh_off ? reinterpret_cast<double*>(ws + fh_off) : nullptr;
  float4* pf = fh_off ? reinterpret_cast<float4*>(ws + pf_off) : nullptr;
  unsigned* count = reinterpret_cast<unsigned*>(ws + alpha_off + kPendingCountOffset);
  if (cudaMemsetAsync(alpha, 0, kAlphaAndCountBytes, st) != cudaSuccess) return TENO_ERR_CUDA;
  if (launch_cell(g->ndim, U, aux, fh, pf, alpha, status, G.ncell, g->gamma, nsm, st, cand) != cudaSuccess)
    return TENO_ERR_CUDA;
  for (int d = 0; d < g->ndim; ++d) {
    if (launch_flux(g->ndim, d, U, aux, fh, pf, alpha, Fhat, nullptr, list, count + d, status, G, S, nsm, st,
                    nullptr, roe_out ? roe_out + d * roe_stride : nullptr) != cudaSuccess)
      return TENO_ERR_CUDA;
    if (launch_diff(g->ndim, d, Fhat, R, Un, Uk, Uout, dt, G, mode, nsm, st, U) != cudaSuccess)
      return TENO_ERR_CUDA;
  }
  return TENO_OK;
}

}  // namespace teno
