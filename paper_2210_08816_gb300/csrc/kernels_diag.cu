// Flow diagnostics of Section 4.2.3: the total kinetic energy (Eq. 12) and the Nusselt number at the hot
// wall (Eq. 13), summed on the device for the time stepper's histories.
//
//   E_kin = 1/2 sum over the interior faces of every velocity component of u_f^2 times the face's control
//           volume: the centre spacing along the component's own axis times the cell widths across it;
//   Nu    = sum over the hot wall's cells (j, k) of (T[k][j][0] - 1) / (dx_0 / 2) dy_j dz_k, Eq. 13 as
//           printed (no sign change: conduction gives -1).
// Both use the metric arrays of the handle (idc[d][f] = 1 / centre spacing, idc[d][0] = 2 / dx_0,
// idx[d][c] = 1 / width) and the library's deterministic two-pass reduction (fixed block partials, then
// their sum in a fixed order).  The wall slot of a face-normal velocity holds 0 and adds nothing.
#include <algorithm>

#include "fv_internal.h"
#include "launch.cuh"

namespace fv {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double r = 0.0;
  if (warp == 0) {
    r = (lane < kThreads / 32) ? sh[lane] : 0.0;
    r = warp_sum(r);
  }
  return r;
}

// Blocks 0 .. be - 1: partial sums of u_f^2 V_f / 2 over the x-rows of the three velocity fields, a warp per row.  The
// two x-factors of the control volumes (centre spacings and widths: one over the metrics) are formed once per block,
// the factors across once per row, a lane each for 32 of a warp's rows, so that a face costs two FP64 operations; with
// a division and four products per face the sum was bound by the FP64 pipe, and with a division by the whole warp for every
// row on grids of short rows (16 x 16 x 800: 72 us, now 25; 2 x 300 x 300 420, now 72).  The other blocks: partial sums of the hot-wall
// flux over the ny * nz wall cells.  (64^3, both diagnostics with their sums: four launches, 70 us of kernels; now two, 18.)
__global__ void __launch_bounds__(kThreads) k_diag_partial(Geo<double> g, const double* q, int be,
                                                            double* __restrict__ part) {
  pdl_begin();
  const unsigned ready0 = pdl_wait();
  q += ready0;
  part += ready0;
  __shared__ double vol[2][kMaxN];
  const int nx = g.n[0], ny = g.n[1], rows = g.n[1] * g.n[2];
  double acc = 0.0;
  if ((int)blockIdx.x < be) {
    for (int x = threadIdx.x; x < nx; x += kThreads) {
      vol[0][x] = 1.0 / g.idc[0][x];
      vol[1][x] = 1.0 / g.idx[0][x];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, step = be * (kThreads / 32);
    for (int r0 = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); r0 < 3 * rows; r0 += 32 * step) {
      double across = 0.0;  // lane i: the factor across of the warp's i-th row from r0 on
      const int mine = r0 + lane * step;
      if (mine < 3 * rows) {
        const int c = mine / rows, jk = mine - c * rows, k = jk / ny, j = jk - k * ny;
        across = 0.5 / ((c == 1 ? g.idc[1][j] : g.idx[1][j]) * (c == 2 ? g.idc[2][k] : g.idx[2][k]));
      }
      for (int i = 0, r = r0; i < 32 && r < 3 * rows; ++i, r += step) {
        const double* f = q + (size_t)r * nx;
        const double* v = vol[r < rows ? 0 : 1];
        double sum = 0.0;
        for (int x = lane; x < nx; x += 32) {
          const double u = f[x];
          sum = fma(u * u, v[x], sum);
        }
        acc = fma(sum, __shfl_sync(0xffffffffu, across, i), acc);
      }
    }
  } else {
    const double* T = q + 3 * (size_t)rows * nx;
    const int bn = gridDim.x - be;
    for (int t = (blockIdx.x - be) * kThreads + threadIdx.x; t < rows; t += bn * kThreads) {
      const int k = t / ny, j = t - k * ny;
      const double grad = (T[(size_t)t * nx] - 1.0) * g.idc[0][0];  // over the half cell dx_0 / 2
      acc += grad / (g.idx[1][j] * g.idx[2][k]);
    }
  }
  const double r = block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = r;
}

// out[0] = sum of part[0 .. be), out[1] = sum of part[be .. be + bn), in a fixed order
__global__ void __launch_bounds__(kThreads) k_diag_finish(const double* part, int be, int bn,
                                                           double* __restrict__ out) {
  pdl_begin();
  const unsigned ready0 = pdl_wait();
  part += ready0;
  out += ready0;
  const double* p = part + (blockIdx.x == 0 ? 0 : be);
  const int n = blockIdx.x == 0 ? be : bn;
  double v = 0.0;
  for (int t = threadIdx.x; t < n; t += kThreads) v += p[t];
  const double r = block_sum(v);
  if (threadIdx.x == 0) out[blockIdx.x] = r;
}

}  // namespace

// E_kin into scalars[slot], Nu into scalars[slot + 1]: one launch for the partials of both, one for the sums
int launch_diagnostics(const fv_grid_s* g, const double* q, int slot) {
  ProfScope ps(g, PROF_REDUCE);
  const int be = std::min(kReduceBlocks, (3 * g->ny * g->nz + 31) / 32);  // four rows per warp
  const int bn = std::min(kReduceBlocks, (g->ny * g->nz + kThreads - 1) / kThreads);
  launch(k_diag_partial, be + bn, kThreads, 0, g->stream, g->geo64, q, be, g->ws.partials);
  FV_CUDA(cudaGetLastError());
  launch(k_diag_finish, 2, kThreads, 0, g->stream, g->ws.partials, be, bn, g->ws.scalars + slot);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

}  // namespace fv
