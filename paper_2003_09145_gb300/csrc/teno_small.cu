// teno_small.cu -- one SSP-RK3 step of a small 1D grid in one launch.
//
// A 1D step of a few hundred to some thousand cells is bound by latency: the
// launch-per-pass path runs 16 dependent kernels, each a few microseconds long
// however small, on a few SMs.  Here one thread-block cluster of up to 16
// CTAs takes the whole step.  Every CTA owns a contiguous range of cells; per
// stage it runs
//   (A) the cell pass of its cells and its maxima of the wave speeds; cluster
//       barrier; the maxima of all CTAs by distributed shared memory; in stage
//       1 the CFL step;
//   (B) its interfaces tile by tile -- the closed form, the open
//       reconstructions, the fluxes of a tile in shared memory -- and the
//       difference fused with the stage; cluster barrier (the next stage's
//       cell pass overwrites what the neighbours read).
// The arithmetic is the launch-per-pass path's, function by function, so the
// results agree bit for bit.
//
// Range of sizes: an FP64 instruction holds an SM partition for 64 cycles per
// warp, so 16 CTAs fall behind 152 SMs once a partition has many warps.
// Measured, us per step, one launch against one per pass, on a smooth tube and on a
// Mach-3 shock into waves (plain calls; in brackets inside a CUDA graph):
//     200 cells   54 / 100 (49 / 78)     68 / 159 (63 / 138)
//    4096         65 / 107 (58 / 84)     78 / 160 (72 / 134)
//    6144         81 / 107 (76 / 84)    113 / 120 (107 / 97)
//    8192         92 / 107 (86 / 84)    130 / 121 (124 / 98)
//   16384        135 / 108 (129 / 84)   228 / 114 (222 / 89)
// so the line is drawn at 16 CTAs of 384 cells.
#include <atomic>
#include <cmath>
#include <cooperative_groups.h>
#include <cstdint>
#include <cuda_runtime.h>

#include "teno.h"
#include "teno_closed.cuh"
#include "teno_device.cuh"
#include "teno_flux.cuh"
#include "teno_launch.h"

namespace teno {

namespace {

namespace cg = cooperative_groups;

constexpr int kSmallThreads = 384;       // most threads per CTA
constexpr int kSmallCtas = 16;           // most CTAs of the cluster
constexpr int kCorrectWarps = 8;         // warps that take open faces

// The stencil of face f: cells f-3 .. f+2, mirrored or virtual beyond the ends.
template <int WALL>
__device__ __forceinline__ void face_cells(const Grid& G, int64_t f, uint32_t (&cells)[6], unsigned& flips) {
  flips = 0u;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const int64_t k = f - 3 + j;
    if (WALL == 2 && (k < 0 || k >= G.n[0])) {
      cells[j] = static_cast<uint32_t>(G.ncell) + (k >= G.n[0]);
    } else {
      bool m;
      cells[j] = static_cast<uint32_t>(ghost(k, G.n[0], G.bc[0], m));
      flips |= unsigned(m) << j;
    }
  }
}

// WALL as in flux_closed_kernel: 1 reflecting, 2 fixed-state faces, 0 neither.
template <int WALL>
__global__ void __launch_bounds__(kSmallThreads) step1d_kernel(SmallStep A, Grid G, Scheme S) {
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ unsigned long long s_red[kSmallThreads / 32][3], s_max[3];
  __shared__ double s_a[3], s_dt;
  __shared__ double s_F[kSmallThreads][3];
  __shared__ int s_pend[kSmallThreads];
  __shared__ int s_npend;
  __shared__ CorrectScratch<1> s_cor[kCorrectWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = blockDim.x, nw = nt >> 5;
  const int64_t n = G.ncell;
  const unsigned rank = cluster.block_rank(), ncta = cluster.num_blocks();
  const int64_t per = (n + ncta - 1) / ncta;
  const int64_t c0 = rank * per < n ? rank * per : n, c1 = c0 + per < n ? c0 + per : n;
  const GhostCells gc{G.gU, G.gaux, G.gfh, G.gpf};
  const double t0 = *A.t;   // before the first barrier: rank 0 writes it after
  double dt = 0.0;
  for (int stage = 0; stage < 3; ++stage) {
    const double* Uin = stage == 0 ? A.U : (stage == 1 ? A.U1 : A.U2);
    double* Uout = stage == 0 ? A.U1 : (stage == 1 ? A.U2 : A.U);
    // (A)
    unsigned long long b0 = 0ull, b1 = 0ull, b2 = 0ull;
    bool bad = false;
    for (int64_t c = c0 + tid; c < c1; c += nt) {
      double uh[1], ep, p, hr, cs;
      if (!cell_primitives<1>(Uin, n, c, S.gamma, A.aux, uh, ep, p, hr)) bad = true;
      if (!sound_speed(p, hr, S.gamma, cs)) bad = true;
      const double Uc[3] = {Uin[c], Uin[n + c], Uin[2 * n + c]};
      const double ph = A.aux[n + c];
      double Fh[3];
      cell_flux_half_ep<1, 0>(Uc, uh[0], ph, ep, Fh);
      A.fh[c] = Fh[1];
      A.fh[n + c] = Fh[2];
      const double su[1] = {A.aux[4 * n + c]};
      store_planes<1>(A.pf, n, c, Uc, uh, ph, A.aux[2 * n + c], A.aux[3 * n + c], su);
      b0 = max_abs_bits(b0, fma(2.0, uh[0], -cs));
      b1 = max_abs_bits(b1, uh[0]);
      b2 = max_abs_bits(b2, fma(2.0, uh[0], cs));
    }
    b1 = dbits(2.0 * __longlong_as_double(static_cast<long long>(b1)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long w0 = __shfl_xor_sync(0xffffffffu, b0, o);
      const unsigned long long w1 = __shfl_xor_sync(0xffffffffu, b1, o);
      const unsigned long long w2 = __shfl_xor_sync(0xffffffffu, b2, o);
      b0 = b0 > w0 ? b0 : w0;
      b1 = b1 > w1 ? b1 : w1;
      b2 = b2 > w2 ? b2 : w2;
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(A.status, kStatusNonphysical);
    if (lane == 0) {
      s_red[warp][0] = b0;
      s_red[warp][1] = b1;
      s_red[warp][2] = b2;
    }
    __syncthreads();
    if (tid < 3) {
      unsigned long long m = 0ull;
      for (int w = 0; w < nw; ++w) m = m > s_red[w][tid] ? m : s_red[w][tid];
      s_max[tid] = m;
    }
    cluster.sync();
    if (warp == 0) {   // lane r reads CTA r's maxima
      unsigned long long m[3];
#pragma unroll
      for (int s = 0; s < 3; ++s) m[s] = lane < int(ncta) ? *cluster.map_shared_rank(&s_max[s], lane) : 0ull;
#pragma unroll
      for (int o = kSmallCtas / 2; o > 0; o >>= 1)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const unsigned long long x = __shfl_xor_sync(0xffffffffu, m[s], o);
          m[s] = m[s] > x ? m[s] : x;
        }
      if (lane < 3) {
        const unsigned long long x = lane == 0 ? m[0] : (lane == 1 ? m[1] : m[2]);
        s_red[0][lane] = x;
        s_a[lane] = 0.5 * __longlong_as_double(static_cast<long long>(x));
        if (rank == 0) A.alpha[lane] = x;
      }
    }
    __syncthreads();
    if (stage == 0) {
      if (tid == 0) {
        // dt_kernel<1>'s step
        const unsigned long long a = s_red[0][0], b = s_red[0][2];
        const double smax = __longlong_as_double(static_cast<long long>(a > b ? a : b));
        double h = A.dt_fixed > 0.0 ? A.dt_fixed : A.cfl * G.dx[0] / smax;
        const double rem = A.t_end - t0;
        if (rem < h) h = rem;
        if (!(h > 0.0)) h = 0.0;
        s_dt = h;
        if (rank == 0) {
          *A.dt_ws = h;
          if (A.dt_out) *A.dt_out = h;
          *A.t = t0 + h;
        }
      }
      __syncthreads();
      dt = s_dt;
      if (!(dt > 0.0)) {
        // t >= t_end: the state stays, the stage buffers take it
        for (int64_t c = c0 + tid; c < c1; c += nt)
#pragma unroll
          for (int v = 0; v < 3; ++v) A.U1[v * n + c] = A.U2[v * n + c] = A.U[v * n + c];
        cluster.sync();   // no CTA leaves while another reads its maxima
        return;
      }
    }
    // (B)
    const double a3[3] = {s_a[0], s_a[1], s_a[2]};
    const FaceSpeeds F = face_speeds(a3);
    const double coef = dt * (G.inv_dx[0] / kFluxScale);
    for (int64_t i0 = c0; i0 < c1; i0 += nt - 1) {
      if (tid == 0) s_npend = 0;
      __syncthreads();
      const int64_t left = c1 - i0 < nt - 1 ? c1 - i0 : nt - 1;   // cells of this tile
      if (tid <= left) {
        uint32_t cells[6];
        unsigned flips;
        face_cells<WALL>(G, i0 + tid, cells, flips);
        double out[3];
        const unsigned open = interface_flux_closed<1, 0, WALL == 2>(
            Uin, A.aux, A.fh, A.pf, n, cells, WALL == 1 ? flips : 0u, a3, F, S, out, A.status, gc);
        if (!(open & kRough)) {
          s_F[tid][0] = out[0];
          s_F[tid][1] = out[1];
          s_F[tid][2] = out[2];
        }
        if (open) s_pend[atomicAdd(&s_npend, 1)] = int(unsigned(tid) | open << 16);
      }
      __syncthreads();
      const int npend = s_npend;
      const int cw = nw < kCorrectWarps ? nw : kCorrectWarps;
      int per_warp = 2;
      while (per_warp < 32 && npend > per_warp * cw) per_warp *= 2;
      auto cells_of = [&](uint32_t f, uint32_t (&cells)[6], unsigned& flips) {
        face_cells<WALL>(G, i0 + f, cells, flips);
        if (WALL != 1) flips = 0u;
      };
      if (warp < cw)
        for (int k0 = warp * per_warp; k0 < npend; k0 += cw * per_warp) {
          const bool mine = lane < per_warp && k0 + lane < npend;
          const unsigned e = mine ? unsigned(s_pend[k0 + lane]) : 0u;
          const int t = int(e & 0xffffu);
          double out[3] = {s_F[t][0], s_F[t][1], s_F[t][2]};
          const double alpha[3] = {a3[0], a3[1], a3[2]};
          warp_correct<1, 0, WALL == 2, uint32_t>(Uin, A.aux, n, cells_of, unsigned(t), alpha, S, e >> 16, out,
                                                  A.status, s_cor[warp], gc);
          if (mine) {
            s_F[t][0] = out[0];
            s_F[t][1] = out[1];
            s_F[t][2] = out[2];
          }
        }
      __syncthreads();
      if (tid < left) {
        const int64_t c = i0 + tid;
        double s[3];
#pragma unroll
        for (int v = 0; v < 3; ++v) s[v] = s_F[tid][v] - s_F[tid + 1][v];
        if (G.has_grav) {   // diff_kernel's source
          const double r = Uin[c] * G.grav[0], w = fma(Uin[n + c], G.grav[0], 0.0);
          s[1] = fma(kFluxScale * G.dx[0], r, s[1]);
          s[2] = fma(kFluxScale * G.dx[0], w, s[2]);
        }
#pragma unroll
        for (int v = 0; v < 3; ++v) Uout[v * n + c] = stage_value(2 + stage, coef, s[v], A.U, Uin, v * n + c);
      }
      __syncthreads();
    }
    cluster.sync();
  }
}

}  // namespace

namespace {

struct SmallShape {
  unsigned ctas, threads;
};
// one warp per SM partition (127 cells a CTA) while 16 CTAs last, then equal
// shares in as few tiles as 384 threads allow
SmallShape small_shape(int64_t n) {
  int64_t ctas = (n + 126) / 127;
  if (ctas > kSmallCtas) ctas = kSmallCtas;
  const int64_t per = (n + ctas - 1) / ctas;
  const int64_t tiles = (per + kSmallThreads - 2) / (kSmallThreads - 1);
  int threads = int(((per + tiles - 1) / tiles + 1 + 31) / 32 * 32);
  if (threads > kSmallThreads) threads = kSmallThreads;
  return {unsigned(ctas), unsigned(threads)};
}

using SmallKernel = void (*)(SmallStep, Grid, Scheme);
// 0 plain, 1 reflecting, 2 fixed-state faces
int small_wall(const Grid& G) { return G.bc[0] == TENO_BC_REFLECTIVE ? 1 : (G.bc[0] == TENO_BC_DIRICHLET ? 2 : 0); }
SmallKernel small_kernel(int wall) {
  return wall == 1 ? step1d_kernel<1> : (wall == 2 ? step1d_kernel<2> : step1d_kernel<0>);
}

struct SmallLaunch {   // (the attribute is referred to by address)
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  SmallLaunch(SmallShape s, cudaStream_t st) {
    cfg.gridDim = dim3(s.ctas);
    cfg.blockDim = dim3(s.threads);
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = s.ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
};

// Whether the current device can hold the cluster at all (more than eight CTAs
// are beyond the portable size, and a device or context with few SMs may not
// schedule them together).  Asked once per device, kernel and shape.
bool cluster_fits(int wall, SmallShape s) {
  static std::atomic<signed char> known[64][3][kSmallCtas + 1][kSmallThreads / 32 + 1];   // 0 not asked, 1, -1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::atomic<signed char>* k = dev < 64 ? &known[dev][wall][s.ctas][s.threads / 32] : nullptr;
  if (k && k->load(std::memory_order_relaxed)) return k->load(std::memory_order_relaxed) > 0;
  const SmallKernel f = small_kernel(wall);
  const SmallLaunch l(s, nullptr);
  int n = 0;
  const bool ok = (s.ctas <= 8 ||
                   cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
                  cudaOccupancyMaxActiveClusters(&n, f, &l.cfg) == cudaSuccess && n > 0;
  if (!ok) cudaGetLastError();   // no error of the step: it takes a launch per pass
  if (k) k->store(ok ? 1 : -1, std::memory_order_relaxed);
  return ok;
}

}  // namespace

// (ndim, not the extents: a 2D or 3D grid of one cell across still has the
// other momenta and their directions' speeds)
bool small_step_applies(int ndim, const Grid& G, const Scheme& S) {
  return ndim == 1 && G.ncell <= kSmallStepMax && S.variant != kSchemeWenoZ &&
         cluster_fits(small_wall(G), small_shape(G.ncell));
}

cudaError_t launch_step1d(const SmallStep& A, const Grid& G, const Scheme& S, cudaStream_t st) {
  const SmallLaunch l(small_shape(G.ncell), st);
  return cudaLaunchKernelEx(&l.cfg, small_kernel(small_wall(G)), A, G, S);
}

}  // namespace teno
