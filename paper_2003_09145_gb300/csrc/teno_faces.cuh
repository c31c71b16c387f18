// teno_faces.cuh -- the grid path's closed-form pass over the interfaces of one
// direction: interface geometry and the loop that the per-direction kernel
// (teno_kernels.cu) and the all-directions one (teno_closed_all.cu) share.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "teno.h"
#include "teno_closed.cuh"
#include "teno_device.cuh"
#include "teno_flux.cuh"

namespace teno {

// ---------------------------------------------------------------------------
// The same fluxes in two passes (no flags).  flux_closed_kernel evaluates the
// closed form with every stencil kept, and its certified FP32 test; the
// interfaces with reconstructions that the test does not prove to be kept go
// to `list` with the mask of those (one atomic per warp), and
// flux_correct_kernel adds their differences (warp_correct).  The
// closed-form pass stays small (registers, instruction cache) and its warps do
// not diverge into the rare slow path, as they do in the one-pass kernel.
// WENO-Z, which keeps no stencil exactly linear, takes flux_wenoz_kernel: the
// characteristic path at every interface, no list.
// ---------------------------------------------------------------------------
#ifndef TENO_CLOSED_MINBLOCKS
#define TENO_CLOSED_MINBLOCKS 4
#endif
// the z sweep's tiled order (below): 36.93 against 37.36 ms per 256^3 RK3 step
#ifndef TENO_CLOSED_Z_TILE
#define TENO_CLOSED_Z_TILE 1
#endif

// The stencil of interface q (32-bit indices throughout: the C-ABI admits
// fewer than 2^32 interfaces per direction).  GH: fixed-state faces along
// DIR, whose ghost points are the virtual cells ncell + 2 DIR + side.
// Interfaces three cells off both ends, nearly all, skip the boundary maps.
template <int NDIM, int DIR, bool GH = false>
__device__ __forceinline__ void interface_cells(uint32_t q, const Grid& G, uint32_t (&cells)[6], unsigned& flips) {
  const uint32_t n0 = static_cast<uint32_t>(G.n[0]), n1 = static_cast<uint32_t>(G.n[1]);
  const uint32_t nd = static_cast<uint32_t>(G.n[DIR]);
  const uint32_t m0 = n0 + (DIR == 0), m1 = n1 + (DIR == 1);
  const uint32_t sd = (DIR == 0) ? 1u : (DIR == 1 ? n0 : n0 * n1);
  uint32_t i0 = q, i1 = 0, i2 = 0;
  if (NDIM > 1) {
    const uint32_t r = q / m0;
    i0 = q - r * m0;
    i1 = r;
    if (NDIM > 2) {
      i2 = r / m1;
      i1 = r - i2 * m1;
    }
  }
  const uint32_t id = (DIR == 0) ? i0 : (DIR == 1 ? i1 : i2);
  const uint32_t base = (DIR == 0) ? (i2 * n1 + i1) * n0 : (DIR == 1) ? i2 * n1 * n0 + i0 : i1 * n0 + i0;
  flips = 0u;
  if (id >= 3u && nd - id >= 3u) {
#pragma unroll
    for (int j = 0; j < 6; ++j) cells[j] = base + (id - 3u + j) * sd;
    return;
  }
  const int bc = G.bc[DIR];
  if (!GH && bc < 2 && nd >= 6u && nd <= 0x7FFFFFF0u) {
    // periodic or zero-gradient ends of lines that a stencil wraps at most
    // once (in the x sweep two warps of five come here at 160 cells a line;
    // the general map's loops and divisions cost them instruction fetches:
    // 21.51 against 21.15 ms per 256^3 step)
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const int k = static_cast<int>(id) - 3 + j, n = static_cast<int>(nd);
      const int w = bc == 0 ? (k < 0 ? k + n : (k >= n ? k - n : k)) : (k < 0 ? 0 : (k >= n ? n - 1 : k));
      cells[j] = base + static_cast<uint32_t>(w) * sd;
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const int64_t k = (int64_t)id - 3 + j;
    if (GH && (k < 0 || k >= (int64_t)nd)) {
      cells[j] = static_cast<uint32_t>(G.ncell) + 2 * DIR + (k >= (int64_t)nd);
    } else {
      bool f;
      cells[j] = base + static_cast<uint32_t>(ghost(k, G.n[DIR], G.bc[DIR], f)) * sd;
      flips |= unsigned(f) << j;
    }
  }
}

template <int NDIM, int DIR>
__device__ __forceinline__ void half_speeds(const unsigned long long* __restrict__ alpha_bits,
                                            double (&alpha)[NDIM + 2], double (&nal)[NDIM + 2]) {
  constexpr int NVAR = NDIM + 2;
  const double am = __longlong_as_double((long long)alpha_bits[DIR * 3 + 0]);
  const double a0 = __longlong_as_double((long long)alpha_bits[DIR * 3 + 1]);
  const double ap = __longlong_as_double((long long)alpha_bits[DIR * 3 + 2]);
  alpha[0] = 0.5 * am;
#pragma unroll
  for (int f = 1; f < NVAR - 1; ++f) alpha[f] = 0.5 * a0;
  alpha[NVAR - 1] = 0.5 * ap;
#pragma unroll
  for (int f = 0; f < NVAR; ++f) nal[f] = -2.0 * alpha[f];
}

// WALL: 1 -- the sweep direction has a reflecting wall, so stencil points may
// be mirrored; 2 -- fixed-state faces (ghost points read from the ghost
// block); 0 -- neither: the mirror flags are the constant 0 and their sign
// flips fold away; 3 -- whichever the grid has (the launch over all directions).
// With ROE every interface's Roe state (the fields that the adjoint's closed-form
// VJP reads: u~, |u~|^2, H~, c~, b1, b1/2, b2/2, 1/(2c~)) and the certificate's
// mask (0: every stencil kept) also go to roe_out[ndim + 8][nifc], for the
// adjoint of this stage.  PF: with the cells' binary32 planes; without them (the largest grids)
// the list holds indices alone, its reconstructions all count as open, and a
// face whose flux stays unwritten (kRough) is marked by a NaN.
template <int NDIM, int DIR, int WALL, bool ROE, bool PF = true, class Entry = uint2>
__device__ __forceinline__ void closed_faces(
    const double* __restrict__ U, const double* __restrict__ aux, const double* __restrict__ fh,
    const float4* __restrict__ pf, const unsigned long long* __restrict__ alpha_bits, double* __restrict__ Fhat,
    Entry* __restrict__ list, unsigned* __restrict__ count, int* __restrict__ status, const Grid& G,
    const Scheme& S, double* __restrict__ roe_out) {
  constexpr int NVAR = NDIM + 2;
  const int64_t nifc = (G.n[0] + (DIR == 0)) * (G.n[1] + (DIR == 1)) * (G.n[2] + (DIR == 2));
  double a3[3];
#pragma unroll
  for (int s = 0; s < 3; ++s) a3[s] = 0.5 * __longlong_as_double((long long)alpha_bits[DIR * 3 + s]);
  const FaceSpeeds F = face_speeds(a3);
  const unsigned lane = threadIdx.x & 31u;
  // The z sweep takes its interfaces in tiles of 32 along x by 4 along z
  // (a block of 128 threads per tile, a warp per z): the six stencil planes
  // of one interface lie a power of two of bytes apart and share L1 sets,
  // so the second pass's reload misses L1 unless the block's four warps
  // read overlapping planes.  The loop runs over whole tiles; lanes past the
  // grid's edge skip.
  constexpr bool ZT = TENO_CLOSED_Z_TILE && DIR == 2 && NDIM == 3;
  const uint32_t n0 = static_cast<uint32_t>(G.n[0]), n1 = static_cast<uint32_t>(G.n[1]);
  const uint32_t nz1 = static_cast<uint32_t>(G.n[2] + 1);
  constexpr uint32_t tx = 32, tz = 4;   // (16 by 8: 21.38 against 21.15 ms per 256^3 step, 8 by 16: 21.46)
  const uint32_t ntx = (n0 + tx - 1u) / tx;
  const int64_t nq = ZT ? (int64_t)ntx * n1 * ((nz1 + tz - 1u) / tz) * 128 : nifc;
  for (int64_t qq = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; qq < nq;
       qq += (int64_t)gridDim.x * blockDim.x) {
    int64_t q = qq;
    if constexpr (ZT) {
      const uint32_t t = static_cast<uint32_t>(qq >> 7), l = static_cast<uint32_t>(qq) & 127u;
      const uint32_t x = (t % ntx) * tx + l % tx;
      const uint32_t r = t / ntx;
      const uint32_t z = (r / n1) * tz + l / tx;
      if (x >= n0 || z >= nz1) continue;
      q = ((int64_t)z * n1 + (r % n1)) * n0 + x;
    }
    uint32_t cells[6];
    unsigned flips;
    if (WALL == 2 || (WALL == 3 && G.bc[DIR] == TENO_BC_DIRICHLET))
      interface_cells<NDIM, DIR, true>(static_cast<uint32_t>(q), G, cells, flips);
    else
      interface_cells<NDIM, DIR, false>(static_cast<uint32_t>(q), G, cells, flips);
    double out[NVAR];
    const unsigned open = interface_flux_closed<NDIM, DIR, (WALL >= 2), PF>(
        U, aux, fh + (int64_t)DIR * (NVAR - 1) * G.ncell, pf, G.ncell, cells, WALL & 1 ? flips : 0u, a3, F, S, out,
        status, GhostCells{G.gU, G.gaux, G.gfh, G.gpf});
    if constexpr (ROE) {
      if (S.keep_idx >= 0) {
        RoeIfc<NDIM> R;
        double su2[NDIM], su3[NDIM];
#pragma unroll
        for (int k = 0; k < NDIM; ++k) {
          su2[k] = aux[(NDIM + 3 + k) * G.ncell + cells[2]];
          su3[k] = aux[(NDIM + 3 + k) * G.ncell + cells[3]];
        }
        roe_interface<NDIM, DIR>(aux[(NDIM + 1) * G.ncell + cells[2]], aux[(NDIM + 1) * G.ncell + cells[3]],
                                 aux[(NDIM + 2) * G.ncell + cells[2]], aux[(NDIM + 2) * G.ncell + cells[3]], su2, su3,
                                 S, R, status);
#pragma unroll
        for (int k = 0; k < NDIM; ++k) roe_out[(int64_t)k * nifc + q] = R.u[k];
        roe_out[(int64_t)(NDIM + 0) * nifc + q] = R.q2;
        roe_out[(int64_t)(NDIM + 1) * nifc + q] = R.H;
        roe_out[(int64_t)(NDIM + 2) * nifc + q] = R.cs;
        roe_out[(int64_t)(NDIM + 3) * nifc + q] = R.b1;
        roe_out[(int64_t)(NDIM + 4) * nifc + q] = R.hb1;
        roe_out[(int64_t)(NDIM + 5) * nifc + q] = R.hb2;
        roe_out[(int64_t)(NDIM + 6) * nifc + q] = R.hic;
        roe_out[(int64_t)(NDIM + 7) * nifc + q] = double(open);
      }
    }
    if constexpr (!PF) {
      if (open & kRough)
#pragma unroll
        for (int v = 0; v < NVAR; ++v) out[v] = __longlong_as_double(0x7FF8000000000000ll);
    }
    if (!PF || !(open & kRough)) {
#pragma unroll
      for (int v = 0; v < NVAR; ++v) Fhat[(int64_t)v * nifc + q] = out[v];
    }
    // append the open interfaces of the lanes converged here
    const unsigned act = __activemask();
    const unsigned m = __ballot_sync(act, open != 0u);
    if (m) {
      const unsigned leader = __ffs(act) - 1;
      unsigned at = 0;
      if (lane == leader) at = atomicAdd(count, __popc(m));
      at = __shfl_sync(act, at, leader);
      if (open) {
        Entry& e = list[at + __popc(m & ((1u << lane) - 1u))];
        if constexpr (PF) e = make_uint2(static_cast<uint32_t>(q), open);
        else e = static_cast<uint32_t>(q);
      }
    }
  }
}

// An FP64 instruction holds its SM partition's pipe for 64 cycles whatever
// lanes are active, so a warp's time is its FP64 instruction count.  A warp
// takes 32 listed interfaces when there are enough for every partition of
// the chip, and fewer (2, 4, 8, 16) when the list is short: a short list is
// bound by one warp's chain, and few interfaces finish in a single round.
template <int NDIM, int DIR, bool GH, class Entry>
__device__ __forceinline__ void correct_list(const double* __restrict__ U, const double* __restrict__ aux,
                                             const unsigned long long* __restrict__ alpha_bits,
                                             double* __restrict__ Fhat, const Entry* __restrict__ list, int64_t n,
                                             int* __restrict__ status, const Grid& G, const Scheme& S, int nsm,
                                             CorrectScratch<NDIM>& W) {
  constexpr int NVAR = NDIM + 2;
  const int64_t nifc = (G.n[0] + (DIR == 0)) * (G.n[1] + (DIR == 1)) * (G.n[2] + (DIR == 2));
  const int64_t nw = (int64_t)gridDim.x * 4;
  int per = 2;
  while (per < 32 && n > (int64_t)per * 4 * nsm) per *= 2;
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  if (blockIdx.x * (int64_t)(4 * per) >= n) return;
  double alpha[NVAR], nal[NVAR];
  half_speeds<NDIM, DIR>(alpha_bits, alpha, nal);
  const bool ghost_dir = GH && G.bc[DIR] == TENO_BC_DIRICHLET;
  auto cells_of = [&](uint32_t q, uint32_t (&cells)[6], unsigned& flips) {
    if (ghost_dir) interface_cells<NDIM, DIR, GH>(q, G, cells, flips);
    else interface_cells<NDIM, DIR, false>(q, G, cells, flips);
  };
  for (int64_t i0 = ((int64_t)blockIdx.x * 4 + warp) * per; i0 < n; i0 += nw * per) {
    const int64_t i = i0 + lane;
    uint2 e = make_uint2(0u, 0u);
    if (lane < per && i < n) {
      if constexpr (sizeof(Entry) == sizeof(uint2)) e = list[i];
      else e = make_uint2(list[i], kAllOpen<NDIM>);
    }
    double out[NVAR];
#pragma unroll
    for (int v = 0; v < NVAR; ++v) out[v] = e.y && !(e.y & kRough) ? Fhat[(int64_t)v * nifc + e.x] : 0.0;
    if constexpr (sizeof(Entry) != sizeof(uint2))
      if (e.y && out[0] != out[0]) e.y |= kRough;   // the mark of an unwritten flux
    warp_correct<NDIM, DIR, GH, uint32_t>(U, aux, G.ncell, cells_of, e.x, alpha, S, e.y, out, status, W,
                                          GhostCells{G.gU, G.gaux, G.gfh, G.gpf});
    if (e.y)
#pragma unroll
      for (int v = 0; v < NVAR; ++v) Fhat[(int64_t)v * nifc + e.x] = out[v];
  }
}

}  // namespace teno
