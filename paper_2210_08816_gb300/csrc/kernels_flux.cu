// The FP64 stencils F (residual) and J.v with every flux computed once.
//
// The same discretisation as everywhere (MAC staggering, conservative central fluxes, Form A; Eqs. 1-6).  Written as
// differences of face and edge fluxes (gradient minus convection, one number per face):
//   edge (x_f[i], y_f[j]):  E_xy = <a_v>_x <b_u>_y + <b_v>_x <a_u>_y   (<.>_d: interpolation along d to the edge)
//     it is the convective flux of u through the y-faces and of v through the x-faces: both momentum equations
//     share it; likewise E_xz and E_yz
//   psi_u^y = d_y b_u - E_xy, psi_v^x = d_x b_v - E_xy, ...            (edges)
//   phi_u   = d_x b_u - (a + a')(b + b') / 2                           (cell centres, along the own axis)
//   theta_d = d_d b_T / Pr - (a_d <b_T>_d + b_d <a_T>_d)               (faces)
// and each equation is a sum over the axes of (high flux - low flux) / spacing.  A cell owns the fluxes on its low
// side; the high ones come from its neighbours: from the next plane of the z-march, and through shared memory from
// the threads of the next x and y (the cells past the tile's high edges belong to two halo warps, which compute the
// x or the y fluxes only).  Interpolations of b reuse the gradients' differences, <b> = b - wl (b - b'), one
// operation each (wl + wr = 1; on a wall face the other factor of the flux is zero).  About 104 operations per cell
// for J.v instead of 285 with both sides computed by every cell.  That is what bounds the FP64 form: GB300 issues two
// FP64 operations per clock and SM.
// Measured (J.v, by the form with both sides per cell before / now): 256^3 7.84 / 3.69 ms (the operations alone take
// 2.9 at 1.23 TFLOP/s), 100^3 709 / 257 us; F at 64^3 137 / 62 us.
//
// Wall cases: with homogeneous wall data the formulas hold as they stand when they read zeros (the halo outside the
// domain is zero-filled, the metric arrays hold the wall values: ic[0] = 2 / dx_0, ic[n] = 2 / dx_{n-1}, wl = wr = 0
// on wall faces); T's zero-flux walls have a zero gradient metric.  J.v relies on zero wall slots (a rule of its
// interface); F ignores what the slots hold.
//
// A tile of tx x ty <= 256 cells is marched over a chunk of z-planes; the planes' tiles (with their halo) arrive in
// a three-slot ring, by TMA where rows and sizes allow, else by cp.async.  tx, ty and the chunk are chosen per grid
// (flux_plan): the number of FP64 warp operations on the busiest SM.
#include <algorithm>
#include <cstring>

#include "fv_internal.h"
#include "launch.cuh"
#include "tcgen05.cuh"

namespace fv {
namespace {

constexpr int kFxCells = 256, kFxThreads = kFxCells + 64, kFxRing = 3;
constexpr int kFxTile = 400;  // elements of one array's plane tile, at most

template <typename R>
struct FxArgs {
  Geo<R> g;
  const R *q, *v;
  R* out;
  R Gr, invPr, sigma;
  int N, tx, ty, pw, pl, zc, nch, use_tma;
  int* err;
  long long spins;
};

template <int BYTES>
__device__ __forceinline__ void cp_async_elem(void* dst, const void* src, int src_bytes) {
  static_assert(BYTES == 4 || BYTES == 8, "element size");
  if (BYTES == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes) : "memory");
}

// A value and its low neighbours along x and y
template <typename R>
struct Tri {
  R c, x, y;
};

// MODE 0: F(q) (b = a = q), MODE 1: J(q) v - sigma v (a = q, b = v)
template <typename R, int MODE>
__global__ void __launch_bounds__(kFxThreads, 1)
    k_flux(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmv,
           const __grid_constant__ FxArgs<R> t) {
  constexpr int NA = MODE == 0 ? 4 : 8;
  constexpr int A = 16 / sizeof(R);  // elements of a 16-byte boundary
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar[kFxRing];
  const Geo<R>& g = t.g;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2], N = t.N;
  const int TX = t.tx, TY = t.ty, PW = t.pw, PL = t.pl;
  R* ring = reinterpret_cast<R*>(smem_raw);  // [kFxRing][NA][PL]
  // exchanged low fluxes, two planes deep: x fluxes [4][TY][TX + 1], y fluxes [4][TY + 1][TX]
  const int XP = TY * (TX + 1), YP = (TY + 1) * TX;
  R* exch = ring + kFxRing * NA * PL;
  const int tid = threadIdx.x;
  const int vec = (int)blockIdx.z / t.nch;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY, k0 = ((int)blockIdx.z - vec * t.nch) * t.zc;
  const int kend = min(k0 + t.zc, nz);
  const int pad = 1 + ((i0 - 1) & (A - 1)), xs = i0 - pad;  // the tile starts on a 16-byte boundary
  const R* q = t.q;
  const R* v = t.v + (size_t)vec * 4 * N;
  R* __restrict__ out = t.out + (size_t)vec * 4 * N;
  pdl_begin();

  // roles: cells; warp 8: the row past the tile's high y edge (y fluxes only); warp 9: the column past its high x
  // edge (x fluxes only)
  int tx, ty;
  bool cell = false, dox, doy;
  if (tid < kFxCells) {
    ty = tid / TX;
    tx = tid - ty * TX;
    cell = dox = doy = ty < TY;
  } else if (tid < kFxCells + 32) {
    tx = tid - kFxCells;
    ty = TY;
    dox = false;
    doy = tx < TX;
  } else {
    tx = TX;
    ty = tid - kFxCells - 32;
    doy = false;
    dox = ty < TY;
  }
  const bool live = dox || doy;
  if (!live) tx = ty = 0;
  const int i = min(i0 + tx, nx), j = min(j0 + ty, ny);
  const bool inside = cell && i0 + tx < nx && j0 + ty < ny;
  const int so = (ty + 1) * PW + tx + pad;  // this thread's cell in a plane tile
  // metrics of the low faces and of the cell
  const R wlx = g.wl[0][i], wrx = g.wr[0][i], icx = g.idc[0][i], ixx = g.idx[0][i], ixmx = i >= 1 ? g.idx[0][i - 1] : R(0);
  const R wly = g.wl[1][j], wry = g.wr[1][j], icy = g.idc[1][j], ixy = g.idx[1][j], ixmy = j >= 1 ? g.idx[1][j - 1] : R(0);
  const R cTx = icx * t.invPr, cTy = (j == 0 || j == ny) ? R(0) : icy * t.invPr;

  if (t.use_tma && tid == 0) {
    for (int s = 0; s < kFxRing; ++s) mbar_init(smem_u32(&bar[s]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const unsigned ready0 = pdl_wait();
  q += ready0;
  if (v) v += ready0;
  out += ready0;

  // plane kk goes to slot (kk - k0 + 1) mod 3; planes outside the domain are not copied (they read as zero)
  auto issue = [&](int kk) {
    const bool kin = kk >= 0 && kk < nz && kk <= kend;
    if (kin) {
      R* slot = ring + ((kk - k0 + 1) % kFxRing) * NA * PL;
      if (t.use_tma) {
        if (tid == 0) {
          const uint32_t b = smem_u32(&bar[(kk - k0 + 1) % kFxRing]);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_expect_tx(b, (uint32_t)(NA * PL * sizeof(R)));
          asm volatile(
              "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
              "%5, %6}], [%2];" ::"r"(smem_u32(slot)),
              "l"(reinterpret_cast<uint64_t>(&tmq)), "r"(b), "r"(xs), "r"(j0 - 1), "r"(kk), "r"(0)
              : "memory");
          if (NA == 8)
            asm volatile(
                "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
                "%4, %5, %6}], [%2];" ::"r"(smem_u32(slot + 4 * PL)),
                "l"(reinterpret_cast<uint64_t>(&tmv)), "r"(b), "r"(xs), "r"(j0 - 1), "r"(kk), "r"(4 * vec)
                : "memory");
        }
      } else {  // warp w copies halo rows w, w + 10, ...
        const int hy = TY + 2;
        for (int row = tid / 32; row < NA * hy; row += kFxThreads / 32) {
          const int arr = row / hy, jj = j0 - 1 + row - arr * hy;
          const R* base = arr < 4 ? q + arr * N : v + (arr - 4) * N;
          const bool rin = jj >= 0 && jj < ny;
          for (int hx = tid & 31; hx < TX + 2; hx += 32) {
            const int ii = i0 - 1 + hx;
            const bool in = rin && ii >= 0 && ii < nx;
            cp_async_elem<sizeof(R)>(slot + arr * PL + (row - arr * hy) * PW + pad - 1 + hx,
                                     in ? base + (kk * ny + jj) * nx + ii : base, in ? (int)sizeof(R) : 0);
          }
        }
      }
    }
    if (!t.use_tma) asm volatile("cp.async.commit_group;" ::: "memory");  // one group per plane, empty or not
    return kin;
  };

  R pa[4], pb[4];              // the cell's values one plane below (u, v, w, T)
  R part[4];                   // x and y terms and low z fluxes of the plane below
  R icz_lo = R(0);             // ic_z of the face below
#pragma unroll
  for (int f = 0; f < 4; ++f) pa[f] = pb[f] = part[f] = R(0);
  // use number of a slot = how often it was copied to: planes outside the domain do not count (only -1, the first)
  const int first = max(k0 - 1, 0);
  int issued = first - 1;
  for (int kk = k0 - 1; kk <= k0 + 1; ++kk)
    if (issue(kk)) issued = kk;
  bool ok = true;
  for (int p = k0 - 1; p <= kend; ++p) {
    const bool kin = p >= 0 && p < nz;
    bool ready = true;
    if (t.use_tma) {
      if (kin) {
        const int s = (p - k0 + 1) % kFxRing;
        // earlier copies into this slot: every third plane back to the first one in the domain
        const int uses = (p - k0 + 1) / kFxRing - ((k0 == 0 && s == 0) ? 1 : 0);
        ready = mbar_wait(smem_u32(&bar[s]), (uint32_t)(uses & 1), t.err, 16, t.spins);
      }
    } else {
      asm volatile("cp.async.wait_group 2;" ::: "memory");  // the two planes after p may still be in flight
      __syncthreads();
    }
    const bool last = p == kend;
    R* ex = exch + (p & 1) * 4 * (XP + YP);
    R lox[4], loy[4];  // low fluxes of the four equations
    R zf[4];
    Tri<R> a[4], b[4];
    const R* slot = ring + ((p - k0 + 1) % kFxRing) * NA * PL + so;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      if (kin && live && ready) {
        a[f].c = slot[f * PL];
        a[f].x = slot[f * PL - 1];
        a[f].y = slot[f * PL - PW];
        if (MODE == 1) {
          b[f].c = slot[(4 + f) * PL];
          b[f].x = slot[(4 + f) * PL - 1];
          b[f].y = slot[(4 + f) * PL - PW];
        }
      } else {
        a[f] = Tri<R>{R(0), R(0), R(0)};
        if (MODE == 1) b[f] = Tri<R>{R(0), R(0), R(0)};
      }
    }
    R Txm = a[3].x;  // F: the hot wall's T = 1 in the gradient
    if (MODE == 0) {  // F ignores what the wall slots hold
      if (i == 0) a[0].c = a[0].y = R(0), Txm = R(1);
      if (i <= 1) a[0].x = R(0);
      if (j == 0) a[1].c = a[1].x = R(0);
      if (j <= 1) a[1].y = R(0);
      if (p <= 0) a[2] = Tri<R>{R(0), R(0), R(0)};
#pragma unroll
      for (int f = 0; f < 4; ++f) b[f] = a[f];
    }
    const int pc = min(max(p, 0), nz);
    const R wlz = g.wl[2][pc], wrz = g.wr[2][pc], icz = g.idc[2][pc], ixz = g.idx[2][pc];
    const R ixmz = pc >= 1 ? g.idx[2][pc - 1] : R(0);
    const R dTz = b[3].c - pb[3], Tf = b[3].c - wlz * dTz;  // T on the z-face p (buoyancy)
    if (p >= k0) {
      // edge fluxes on the z-face p, with the differences of b they share with the gradients
      R exz = R(0), eyz = R(0);
      const R duz = b[0].c - pb[0], dvz = b[1].c - pb[1];
      R dwx = R(0), dwy = R(0);
      if (dox) {
        dwx = b[2].c - b[2].x;
        const R aw = wlx * a[2].x + wrx * a[2].c, au = wlz * pa[0] + wrz * a[0].c;
        exz = MODE == 1 ? aw * (b[0].c - wlz * duz) + (b[2].c - wlx * dwx) * au : aw * au;
      }
      if (doy) {
        dwy = b[2].c - b[2].y;
        const R aw = wly * a[2].y + wry * a[2].c, av = wlz * pa[1] + wrz * a[1].c;
        eyz = MODE == 1 ? aw * (b[1].c - wlz * dvz) + (b[2].c - wly * dwy) * av : aw * av;
      }
      if (cell) {  // z fluxes at face p: they close plane p - 1
        const R cTz = (p == 0 || p == nz) ? R(0) : icz * t.invPr;
        zf[0] = duz * icz - exz;
        zf[1] = dvz * icz - eyz;
        if (MODE == 1) {
          zf[2] = (b[2].c - pb[2]) * ixmz - R(0.5) * (a[2].c + pa[2]) * (b[2].c + pb[2]);
          zf[3] = dTz * cTz - (a[2].c * Tf + b[2].c * (wlz * pa[3] + wrz * a[3].c));
        } else {
          const R m = a[2].c + pa[2];
          zf[2] = (b[2].c - pb[2]) * ixmz - R(0.25) * m * m;
          zf[3] = dTz * cTz - a[2].c * Tf;
        }
        if (p > k0 && inside && ready) {
          const int o = ((p - 1) * ny + j) * nx + i;
          out[o] = i >= 1 ? part[0] + zf[0] * ixmz : R(0);
          out[N + o] = j >= 1 ? part[1] + zf[1] * ixmz : R(0);
          out[2 * N + o] = p - 1 >= 1 ? part[2] + zf[2] * icz_lo : R(0);
          out[3 * N + o] = part[3] + zf[3] * ixmz;
        }
      }
      if (!last) {
        const R duy = b[0].c - b[0].y, dvx = b[1].c - b[1].x;
        const R av = wlx * a[1].x + wrx * a[1].c, au = wly * a[0].y + wry * a[0].c;
        const R exy = MODE == 1 ? av * (b[0].c - wly * duy) + (b[1].c - wlx * dvx) * au : av * au;
        if (dox) {
          const R dT = b[3].c - b[3].x;
          if (MODE == 1) {
            lox[0] = (b[0].c - b[0].x) * ixmx - R(0.5) * (a[0].c + a[0].x) * (b[0].c + b[0].x);
            lox[3] = dT * cTx - (a[0].c * (b[3].c - wlx * dT) + b[0].c * (wlx * a[3].x + wrx * a[3].c));
          } else {
            const R m = a[0].c + a[0].x;
            lox[0] = (b[0].c - b[0].x) * ixmx - R(0.25) * m * m;
            lox[3] = (a[3].c - Txm) * cTx - a[0].c * (a[3].c - wlx * dT);
          }
          lox[1] = dvx * icx - exy;
          lox[2] = dwx * icx - exz;
          const int o = ty * (TX + 1) + tx;
#pragma unroll
          for (int f = 0; f < 4; ++f) ex[f * XP + o] = lox[f];
        }
        if (doy) {
          const R dT = b[3].c - b[3].y;
          loy[0] = duy * icy - exy;
          if (MODE == 1) {
            loy[1] = (b[1].c - b[1].y) * ixmy - R(0.5) * (a[1].c + a[1].y) * (b[1].c + b[1].y);
            loy[3] = dT * cTy - (a[1].c * (b[3].c - wly * dT) + b[1].c * (wly * a[3].y + wry * a[3].c));
          } else {
            const R m = a[1].c + a[1].y;
            loy[1] = (b[1].c - b[1].y) * ixmy - R(0.25) * m * m;
            loy[3] = dT * cTy - a[1].c * (b[3].c - wly * dT);
          }
          loy[2] = dwy * icy - eyz;
          const int o = ty * TX + tx;
#pragma unroll
          for (int f = 0; f < 4; ++f) ex[4 * XP + f * YP + o] = loy[f];
        }
      }
    }
    ok = __syncthreads_and(ready);  // fluxes exchanged; nobody reads plane p's slot any more; stop together
    if (!ok) break;
    if (p + 3 <= kend) {
      if (issue(p + 3)) issued = p + 3;
    } else if (!t.use_tma) {
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (p >= k0 && !last && cell) {
      const int ox = ty * (TX + 1) + tx + 1, oy = (ty + 1) * TX + tx;
      R hx[4], hy[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        hx[f] = ex[f * XP + ox] - lox[f];
        hy[f] = ex[4 * XP + f * YP + oy] - loy[f];
      }
      part[0] = hx[0] * icx + hy[0] * ixy - zf[0] * ixz;
      part[1] = hx[1] * ixx + hy[1] * icy - zf[1] * ixz;
      part[2] = hx[2] * ixx + hy[2] * ixy - zf[2] * icz + t.Gr * Tf;
      part[3] = hx[3] * ixx + hy[3] * ixy - zf[3] * ixz;
      if (MODE == 1) {
#pragma unroll
        for (int f = 0; f < 4; ++f) part[f] -= t.sigma * b[f].c;
      }
    }
    icz_lo = icz;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      pa[f] = a[f].c;
      pb[f] = b[f].c;
    }
  }
  // give-up path: every plane copy still in flight lands (waited for with the full limit) before the CTA exits
  if (!ok && t.use_tma && tid == 0)
    for (int kk = max(first, issued - kFxRing + 1); kk <= issued; ++kk) {
      const int s = (kk - k0 + 1) % kFxRing;
      const int uses = (kk - k0 + 1) / kFxRing - ((k0 == 0 && s == 0) ? 1 : 0);
      mbar_wait(smem_u32(&bar[s]), (uint32_t)(uses & 1), t.err, 16, kWaitLimit);
    }
}

// columns of a tile: up to two before the first cell, tx cells, one after; rows on 16-byte boundaries
int tile_width(int tx) { return (tx + 4) / 2 * 2; }

}  // namespace

// Cells per tile and planes per CTA: the fewest FP64 warp operations on the busiest SM (104 per warp of cells and
// plane, 45 of them again for a chunk's closing plane, 40 for each halo warp and plane, and 400 for a CTA's start;
// two operations per clock and SM, so a warp operation takes 16 clocks).  A launch with fewer CTAs than SMs is bound
// by a scheduler's share instead: it takes the warps of a CTA in fours.  The width divides the axis as evenly as it
// can (100 cells: 4 x 25; 32-wide tiles would leave 28 % of the lanes idle).
static FluxPlan flux_plan(const fv_grid_s* g, int nvec) {
  FluxPlan best{};
  double cost = -1.0;
  for (int parts = (g->nx + 31) / 32; parts <= (g->nx + 31) / 32 + 2; ++parts) {
    const int tx = (g->nx + parts - 1) / parts;
    for (int ty = 1; ty <= 16 && tx * ty <= kFxCells; ++ty) {
      const int pl = (ty + 2) * tile_width(tx);
      if (pl > kFxTile) break;
      if ((4 * pl * sizeof(double)) % 128 != 0) continue;  // a state's box of a TMA plane keeps the next one aligned
      const long long tiles = (long long)((g->nx + tx - 1) / tx) * ((g->ny + ty - 1) / ty) * nvec;
      const int warps = (tx * ty + 31) / 32;
      each_chunk(g->nz, [&](int zc, int n) {
        if ((long long)n * nvec > 65535) return false;
        const int w = tiles * n <= g->sms ? (warps + 3) / 4 * 4 : warps;
        const double per = 400.0 + zc * (104.0 * w + 80.0) + 45.0 * w;
        const double c = per * (double)((tiles * n + g->sms - 1) / g->sms);
        if (cost < 0.0 || c < cost) {
          cost = c;
          best = FluxPlan{nvec, tx, ty, zc};
        }
        return true;
      });
    }
  }
  return best;
}

int flux_setup() {
  auto most = [](int arrays) { return (int)((kFxRing * arrays * kFxTile + 8 * (2 * kFxCells + 64)) * sizeof(double)); };
  FV_CUDA(cudaFuncSetAttribute(k_flux<double, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, most(4)));
  FV_CUDA(cudaFuncSetAttribute(k_flux<double, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, most(8)));
  return FV_OK;
}

template <int MODE>
int launch_flux(const fv_grid_s* g, double Gr, double sigma, const double* q, const double* v, double* out, int nvec) {
  using R = double;
  constexpr int NA = MODE == 0 ? 4 : 8;
  FluxPlan& pl = g->flux[nvec > 1];
  if (pl.nvec != nvec) pl = flux_plan(g, nvec);
  if (pl.nvec != nvec) {
    set_error("launch_flux: too many vectors in one block");
    return FV_EINVAL;
  }
  FxArgs<R> t{};
  t.g = g->geo64;
  t.q = q;
  t.v = v;
  t.out = out;
  t.Gr = (R)Gr;
  t.invPr = (R)(1.0 / g->Pr);
  t.sigma = (R)sigma;
  t.N = (int)g->N;
  t.tx = pl.tx;
  t.ty = pl.ty;
  t.zc = pl.zc;
  t.nch = (g->nz + pl.zc - 1) / pl.zc;
  t.pw = tile_width(pl.tx);
  t.err = g->ws.err;
  t.spins = wait_spins(g);
  // TMA: rows and bases on 16-byte boundaries
  t.use_tma = (g->nx * sizeof(R)) % 16 == 0 && (uintptr_t)q % 16 == 0 && (uintptr_t)v % 16 == 0;
  t.pl = (pl.ty + 2) * t.pw;
  CUtensorMap tq, tv;
  std::memset(&tq, 0, sizeof(tq));
  std::memset(&tv, 0, sizeof(tv));
  if (t.use_tma) {
    const uint64_t strides[3] = {g->nx * sizeof(R), (uint64_t)g->nx * g->ny * sizeof(R), g->N * sizeof(R)};
    const uint32_t box[4] = {(uint32_t)t.pw, (uint32_t)pl.ty + 2, 1, 4};
    const CUtensorMapDataType ty = CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
    const uint64_t dq[4] = {(uint64_t)g->nx, (uint64_t)g->ny, (uint64_t)g->nz, 4};
    const uint64_t dv[4] = {(uint64_t)g->nx, (uint64_t)g->ny, (uint64_t)g->nz, 4 * (uint64_t)nvec};
    if (t.use_tma && (encode_tensor_map(&tq, ty, 4, q, dq, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE) != FV_OK ||
                      encode_tensor_map(&tv, ty, 4, v, dv, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE) != FV_OK))
      t.use_tma = 0;
  }
  const size_t smem = ((size_t)kFxRing * NA * t.pl + 8 * ((size_t)pl.ty * (pl.tx + 1) + (size_t)(pl.ty + 1) * pl.tx)) * sizeof(R);
  const dim3 grid((g->nx + pl.tx - 1) / pl.tx, (g->ny + pl.ty - 1) / pl.ty, t.nch * nvec);
  ProfScope ps(g, PROF_STENCIL);
  launch(k_flux<R, MODE>, grid, kFxThreads, smem, g->stream, tq, tv, t);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

template int launch_flux<0>(const fv_grid_s*, double, double, const double*, const double*, double*, int);
template int launch_flux<1>(const fv_grid_s*, double, double, const double*, const double*, double*, int);

}  // namespace fv
