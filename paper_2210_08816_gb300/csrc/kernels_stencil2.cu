// J.v (FP32) with two x-adjacent cells per thread.
//
// The same discretisation as the z-marching stencil of kernels_stencil.cu (MAC staggering, conservative
// central fluxes, Form A; Eqs. 1-2 linearised about q, homogeneous wall data), the same plane ring in
// shared memory filled by 4D TMA boxes, but a thread computes the cells (x, y) and (x + 1, y), x even.
// The two cells share most of their x-neighbours, so the ring is read with 8-byte loads (pairs at even
// offsets) plus scalars (odd offsets): about half the shared-memory loads per cell, the instruction
// stream that bounded the one-cell form.  Block: 64 x 8 cells (256 threads), z-chunks by stencil_chunk.
// Wall cases without branches as in the one-cell J.v form: the face-normal wall slot holds zero, the
// halo outside the domain arrives zero-filled, and the metric arrays hold the wall values; only T's
// zero-flux walls (y, z) are selects.
#include <cstring>

#include "fv_internal.h"
#include "launch.cuh"

namespace fv {
namespace {

constexpr int kPX = 64, kPY = 8, kPHY = kPY + 2;
constexpr int kPW2 = 72;            // ring row: x from i0 - 4 to i0 + 67 (TMA x start on a 16-byte boundary)
constexpr int kPX0 = 4;             // column of the tile's first cell
constexpr int kPL2 = kPHY * kPW2;   // one array's plane tile
constexpr int kPRing = 4, kPNA = 8;
constexpr PlaneTimes kPairTimes = {2, {10, 17, 0}};
constexpr size_t kPairSmem = (size_t)kPRing * kPNA * kPL2 * sizeof(float);
constexpr long long kPWaitLimit = 1LL << 22;

// ---------------------------------------------------------------- pair arithmetic
// Blackwell's packed FP32 instructions (PTX add / sub / mul / fma .rn.f32x2): one instruction per pair,
// the same IEEE round-to-nearest results as the two scalar operations.
__device__ __forceinline__ unsigned long long pk(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 upk(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ float2 operator+(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk(a)), "l"(pk(b)));
  return upk(r);
}
__device__ __forceinline__ float2 operator-(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk(a)), "l"(pk(b)));
  return upk(r);
}
__device__ __forceinline__ float2 operator*(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk(a)), "l"(pk(b)));
  return upk(r);
}
// a * b + c, one rounding
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pk(a)), "l"(pk(b)), "l"(pk(c)));
  return upk(r);
}
__device__ __forceinline__ float2 bc(float s) { return make_float2(s, s); }

// Metric values of one axis as the stencil uses them (cell index c): per pair (float2, x) or per thread
// (float, y and z).
template <typename T>
struct Bundle {
  T ix, ixm, ic, icp, wl, wr, wlp, wrp;
};

__device__ __forceinline__ Bundle<float> load_bundle(const Geo<float>& g, int d, int c) {
  Bundle<float> m;
  const int n = g.n[d];
  m.ix = __ldg(g.idx[d] + c);
  m.ixm = c >= 1 ? __ldg(g.idx[d] + c - 1) : 0.f;
  m.ic = __ldg(g.idc[d] + c);
  m.icp = __ldg(g.idc[d] + c + 1);
  m.wl = __ldg(g.wl[d] + c);
  m.wr = __ldg(g.wr[d] + c);
  m.wlp = c + 1 <= n ? __ldg(g.wl[d] + c + 1) : 0.f;
  m.wrp = c + 1 <= n ? __ldg(g.wr[d] + c + 1) : 0.f;
  return m;
}

__device__ __forceinline__ Bundle<float2> broadcast(const Bundle<float>& a) {
  Bundle<float2> m;
  m.ix = bc(a.ix);
  m.ixm = bc(a.ixm);
  m.ic = bc(a.ic);
  m.icp = bc(a.icp);
  m.wl = bc(a.wl);
  m.wr = bc(a.wr);
  m.wlp = bc(a.wlp);
  m.wrp = bc(a.wrp);
  return m;
}

__device__ __forceinline__ Bundle<float2> load_bundle_pair(const Geo<float>& g, int c) {
  const Bundle<float> a = load_bundle(g, 0, c), b = load_bundle(g, 0, c + 1);
  Bundle<float2> m;
  m.ix = make_float2(a.ix, b.ix);
  m.ixm = make_float2(a.ixm, b.ixm);
  m.ic = make_float2(a.ic, b.ic);
  m.icp = make_float2(a.icp, b.icp);
  m.wl = make_float2(a.wl, b.wl);
  m.wr = make_float2(a.wr, b.wr);
  m.wlp = make_float2(a.wlp, b.wlp);
  m.wrp = make_float2(a.wrp, b.wrp);
  return m;
}

template <int D>
__device__ __forceinline__ decltype(auto) pick(const Bundle<float2>& x, const Bundle<float2>& y, const Bundle<float2>& z) {
  if constexpr (D == 0)
    return (x);
  else if constexpr (D == 1)
    return (y);
  else
    return (z);
}

__host__ __device__ constexpr int unit_(int d, int c) { return d == c ? 1 : 0; }

// The ring seen from one pair: p[dz + 1] points at the pair's first cell in array 0 of plane k + dz.
struct Ring2 {
  const float* p[3];
  template <int A, int DX, int DY, int DZ>
  __device__ __forceinline__ float2 ld() const {
    const float* s = p[DZ + 1] + A * kPL2 + DY * kPW2 + DX;
    if constexpr ((DX & 1) == 0)
      return *reinterpret_cast<const float2*>(s);  // 8-byte aligned: the pair's column is even
    else
      return make_float2(s[0], s[1]);
  }
};


// The convective flux of momentum component C through the low or high D-face of its control volume (D != C): the
// D-velocity interpolated along C to the edge times the C-velocity interpolated along D.  Exchanging C and D exchanges
// the two factors: components C and D share the flux of every edge.  n: the C-pair across the face.
template <int C, int D>
__device__ __forceinline__ float2 edge_lo(const Ring2& S, const Bundle<float2>& MC, const Bundle<float2>& MD, float2 aH,
                                          float2 bH, float2 bCm) {
  constexpr int cx = unit_(C, 0), cy = unit_(C, 1), cz = unit_(C, 2);
  constexpr int dx = unit_(D, 0), dy = unit_(D, 1), dz = unit_(D, 2);
  constexpr int AB = 4;
  const float2 aDc = fma2(MC.wl, S.ld<D, -cx, -cy, -cz>(), MC.wr * S.ld<D, 0, 0, 0>());
  const float2 bDc = fma2(MC.wl, S.ld<AB + D, -cx, -cy, -cz>(), MC.wr * S.ld<AB + D, 0, 0, 0>());
  const float2 aCd = fma2(MD.wl, S.ld<C, -dx, -dy, -dz>(), MD.wr * aH);
  const float2 bCd = fma2(MD.wl, bCm, MD.wr * bH);
  return fma2(aDc, bCd, bDc * aCd);
}
template <int C, int D>
__device__ __forceinline__ float2 edge_hi(const Ring2& S, const Bundle<float2>& MC, const Bundle<float2>& MD, float2 aH,
                                          float2 bH, float2 bCp) {
  constexpr int cx = unit_(C, 0), cy = unit_(C, 1), cz = unit_(C, 2);
  constexpr int dx = unit_(D, 0), dy = unit_(D, 1), dz = unit_(D, 2);
  constexpr int AB = 4;
  const float2 aDc = fma2(MC.wl, S.ld<D, dx - cx, dy - cy, dz - cz>(), MC.wr * S.ld<D, dx, dy, dz>());
  const float2 bDc = fma2(MC.wl, S.ld<AB + D, dx - cx, dy - cy, dz - cz>(), MC.wr * S.ld<AB + D, dx, dy, dz>());
  const float2 aCd = fma2(MD.wlp, aH, MD.wrp * S.ld<C, dx, dy, dz>());
  const float2 bCd = fma2(MD.wlp, bH, MD.wrp * bCp);
  return fma2(aDc, bCd, bDc * aCd);
}

// conv, lap += the share of the D-faces of component C, whose low edge's convective flux is fLo
template <int C, int D>
__device__ __forceinline__ void across(const Ring2& S, const Bundle<float2>& MC, const Bundle<float2>& MD, float2 aH,
                                       float2 bH, float2 fLo, float2& conv, float2& lap) {
  constexpr int dx = unit_(D, 0), dy = unit_(D, 1), dz = unit_(D, 2);
  constexpr int AB = 4;
  const float2 bCm = S.ld<AB + C, -dx, -dy, -dz>(), bCp = S.ld<AB + C, dx, dy, dz>();
  const float2 fHi = edge_hi<C, D>(S, MC, MD, aH, bH, bCp);
  const float2 gLo = (bH - bCm) * MD.ic, gHi = (bCp - bH) * MD.icp;
  conv = fma2(fHi - fLo, MD.ix, conv);
  lap = fma2(gHi - gLo, MD.ix, lap);
}

// the same through the z-faces of u and v: both fluxes of the low face are the plane below's high ones (f, g), which
// become this plane's
template <int C>
__device__ __forceinline__ void across_z(const Ring2& S, const Bundle<float2>& MC, const Bundle<float2>& mz, float2 aH,
                                         float2 bH, float2& f, float2& g, float2& conv, float2& lap) {
  const float2 bCp = S.ld<4 + C, 0, 0, 1>();
  const float2 fHi = edge_hi<C, 2>(S, MC, mz, aH, bH, bCp);
  const float2 gHi = (bCp - bH) * mz.icp;
  conv = fma2(fHi - f, mz.ix, conv);
  lap = fma2(gHi - g, mz.ix, lap);
  f = fHi;
  g = gHi;
}

// conv, lap of component C (x or y) through the faces across its own axis
template <int C>
__device__ __forceinline__ void along(const Ring2& S, const Bundle<float2>& MC, float2 aH, float2 bH, float2& conv,
                                      float2& lap) {
  constexpr int cx = unit_(C, 0), cy = unit_(C, 1);
  const float2 aM = S.ld<C, -cx, -cy, 0>(), bM = S.ld<4 + C, -cx, -cy, 0>();
  const float2 aP = S.ld<C, cx, cy, 0>(), bP = S.ld<4 + C, cx, cy, 0>();
  const float2 half = bc(0.5f), two = bc(2.f);
  const float2 aE = half * (aH + aP), bE = half * (bH + bP);
  const float2 aW = half * (aM + aH), bW = half * (bM + bH);
  conv = two * (aE * bE - aW * bW) * MC.ic;
  lap = ((bP - bH) * MC.ix - (bH - bM) * MC.ixm) * MC.ic;
}

// Fluxes through the low z-faces of a pair's four control volumes (convective f, diffusive g); across the w-face's own
// axis the product of the halved sums and the scaled difference.  A thread marches along z: the next plane's low
// fluxes are this plane's high ones, and w's low x- and y-edges are u's and v's low z-edges.
struct LowZ {
  float2 f[4], g[4];
};

// Temperature fluxes through the D-faces of the cell; y, z walls: zero flux (select), x: Dirichlet 0
template <int D, typename BD>
__device__ __forceinline__ void temperature_dir(const Ring2& S, const BD& MD, float2 TaH, float2 TbH, bool lo_in,
                                                bool hi_in, float2& conv, float2& lap) {
  constexpr int dx = unit_(D, 0), dy = unit_(D, 1), dz = unit_(D, 2);
  constexpr int AB = 4;
  const float2 Tam = S.ld<3, -dx, -dy, -dz>(), Tbm = S.ld<AB + 3, -dx, -dy, -dz>();
  const float2 fLo = fma2(S.ld<D, 0, 0, 0>(), fma2(MD.wl, Tbm, MD.wr * TbH),
                          S.ld<AB + D, 0, 0, 0>() * fma2(MD.wl, Tam, MD.wr * TaH));
  float2 gLo = (TbH - Tbm) * MD.ic;
  const float2 Tap = S.ld<3, dx, dy, dz>(), Tbp = S.ld<AB + 3, dx, dy, dz>();
  const float2 fHi = fma2(S.ld<D, dx, dy, dz>(), fma2(MD.wlp, TbH, MD.wrp * Tbp),
                          S.ld<AB + D, dx, dy, dz>() * fma2(MD.wlp, TaH, MD.wrp * Tap));
  float2 gHi = (Tbp - TbH) * MD.icp;
  if (!lo_in) gLo = make_float2(0.f, 0.f);
  if (!hi_in) gHi = make_float2(0.f, 0.f);
  conv = fma2(fHi - fLo, MD.ix, conv);
  lap = fma2(gHi - gLo, MD.ix, lap);
}

__device__ __forceinline__ void temperature_pair(const Ring2& S, const Bundle<float2>& mx, const Bundle<float2>& my,
                                                 const Bundle<float2>& mz, int j, int ny, int k, int nz, float2& f,
                                                 float2& g, float2& conv, float2& lap) {
  const float2 TaH = S.ld<3, 0, 0, 0>(), TbH = S.ld<4 + 3, 0, 0, 0>();
  conv = make_float2(0.f, 0.f);
  lap = make_float2(0.f, 0.f);
  temperature_dir<0>(S, mx, TaH, TbH, true, true, conv, lap);
  temperature_dir<1>(S, my, TaH, TbH, j >= 1, j + 1 <= ny - 1, conv, lap);
  const float2 Tap = S.ld<3, 0, 0, 1>(), Tbp = S.ld<4 + 3, 0, 0, 1>();
  const float2 fHi = fma2(S.ld<2, 0, 0, 1>(), fma2(mz.wlp, TbH, mz.wrp * Tbp),
                          S.ld<4 + 2, 0, 0, 1>() * fma2(mz.wlp, TaH, mz.wrp * Tap));
  float2 gHi = (Tbp - TbH) * mz.icp;
  if (k + 1 > nz - 1) gHi = make_float2(0.f, 0.f);
  conv = fma2(fHi - f, mz.ix, conv);
  lap = fma2(gHi - g, mz.ix, lap);
  f = fHi;
  g = gHi;
}

__device__ __forceinline__ void low_z(const Ring2& S, const Bundle<float2>& mx, const Bundle<float2>& my,
                                      const Bundle<float2>& mz, int k, LowZ& z) {
  const float2 half = bc(0.5f);
  const float2 bu = S.ld<4, 0, 0, -1>(), bv = S.ld<5, 0, 0, -1>(), bH0 = S.ld<4, 0, 0, 0>(), bH1 = S.ld<5, 0, 0, 0>();
  z.f[0] = edge_lo<0, 2>(S, mx, mz, S.ld<0, 0, 0, 0>(), bH0, bu);
  z.g[0] = (bH0 - bu) * mz.ic;
  z.f[1] = edge_lo<1, 2>(S, my, mz, S.ld<1, 0, 0, 0>(), bH1, bv);
  z.g[1] = (bH1 - bv) * mz.ic;
  const float2 bM = S.ld<6, 0, 0, -1>(), bH2 = S.ld<6, 0, 0, 0>();
  z.f[2] = half * (S.ld<2, 0, 0, -1>() + S.ld<2, 0, 0, 0>()) * (half * (bM + bH2));
  z.g[2] = (bH2 - bM) * mz.ixm;
  const float2 Tam = S.ld<3, 0, 0, -1>(), Tbm = S.ld<7, 0, 0, -1>();
  const float2 TaH = S.ld<3, 0, 0, 0>(), TbH = S.ld<7, 0, 0, 0>();
  z.f[3] = fma2(S.ld<2, 0, 0, 0>(), fma2(mz.wl, Tbm, mz.wr * TbH), bH2 * fma2(mz.wl, Tam, mz.wr * TaH));
  z.g[3] = k >= 1 ? (TbH - Tbm) * mz.ic : make_float2(0.f, 0.f);
}

__device__ __forceinline__ uint32_t smem_addr2(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ bool bar_try2(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait on an mbarrier phase (at most `spins` polls); on expiry records code 17 in *err
__device__ __forceinline__ bool bar_wait2(uint32_t bar, uint32_t parity, int* err, long long spins) {
  for (long long i = 0; i < spins; ++i)
    if (bar_try2(bar, parity)) return true;
  atomicCAS(err, 0, 17);
  return false;
}


// J.v, FP32, two cells per thread; ring planes arrive as one 4D TMA box per state (x, y, z, field)
template <bool BLOCK>
__global__ void __launch_bounds__(kPX / 2 * kPY, 2)
    k_stencil_pair(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmv, int* err,
                   long long spins, Geo<float> g, int N, float Gr, float invPr, float sigma, float* __restrict__ out, int zc,
                   int nch, const TempOut t) {
  constexpr uint32_t kBox = 4u * kPL2 * sizeof(float);  // one state's box: 4 fields x kPHY x kPW2
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar[kPRing], bar_done[2];
  float* sm = reinterpret_cast<float*>(smem_raw);  // [kPRing][kPNA][kPL2]
  const int tid = threadIdx.x;
  const int tx = tid % (kPX / 2), ty = tid / (kPX / 2);
  // BLOCK: blockIdx.z = z-chunk + nch * vector, vector `vec` of the block is fields 4 vec .. 4 vec + 3 of
  // tmv; otherwise one vector in chunks of zc planes
  if (!BLOCK) nch = gridDim.z;
  const int vec = BLOCK ? (int)blockIdx.z / nch : 0;
  const int i0 = blockIdx.x * kPX, j0 = blockIdx.y * kPY, k0 = ((int)blockIdx.z - vec * nch) * zc;
  if (BLOCK) out += (size_t)vec * 4 * N;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const int kend = min(k0 + zc, nz);
  pdl_begin();
  if (tid == 0) {
    for (int s2 = 0; s2 < kPRing; ++s2)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr2(&bar[s2])) : "memory");
    for (int s2 = 0; s2 < 2; ++s2)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr2(&bar_done[s2])), "r"(kPX / 2 * kPY / 32)
                   : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const unsigned ready0 = pdl_wait();
  out += ready0;
  // thread 0: plane kk of both states (zeros outside the domain)
  auto issue_plane = [&](int kk) {
    float* slot = sm + ((kk + kPRing) % kPRing) * kPNA * kPL2;
    const uint32_t b = smem_addr2(&bar[(kk + kPRing) % kPRing]);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(2u * kBox) : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
        "%5, %6}], [%2];" ::"r"(smem_addr2(slot)),
        "l"(reinterpret_cast<uint64_t>(&tmq)), "r"(b), "r"(i0 - kPX0), "r"(j0 - 1), "r"(kk), "r"(0)
        : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
        "%5, %6}], [%2];" ::"r"(smem_addr2(slot + 4 * kPL2)),
        "l"(reinterpret_cast<uint64_t>(&tmv)), "r"(b), "r"(i0 - kPX0), "r"(j0 - 1), "r"(kk), "r"(4 * vec)
        : "memory");
  };
  // plane kk lives in slot kk mod kPRing; it is that slot's use number (kk - k0 + 1) / kPRing
  auto wait_plane = [&](int kk) -> bool {
    return bar_wait2(smem_addr2(&bar[(kk + kPRing) % kPRing]), (uint32_t)(((kk - k0 + 1) / kPRing) & 1), err,
                     spins);
  };
  if (tid == 0)
    for (int kk = k0 - 1; kk <= k0 + 1; ++kk) issue_plane(kk);
  int issued = k0 + 1;  // (thread 0) last plane whose copy was started
  bool ok = wait_plane(k0 - 1);
  ok = wait_plane(k0) && ok;
  ok = __all_sync(0xffffffffu, ok);
  const int x = i0 + 2 * tx, j = j0 + ty;
  const bool active = (x < nx && j < ny);  // nx is a multiple of kPX: both cells are in the domain
  const Bundle<float2> mx = load_bundle_pair(g, active ? x : 0);
  const Bundle<float2> my = broadcast(load_bundle(g, 1, active ? j : 0));
  LowZ z;
  if (active && ok) {
    Ring2 S;
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
      S.p[dz + 1] = sm + ((k0 + dz + kPRing) % kPRing) * kPNA * kPL2 + (ty + 1) * kPW2 + (2 * tx + kPX0);
    low_z(S, mx, my, broadcast(load_bundle(g, 2, k0)), k0, z);
  }
  for (int k = k0; k < kend && ok; ++k) {
    const Bundle<float2> mz = broadcast(load_bundle(g, 2, k));
    const size_t oT = (size_t)(4 * vec + 3) * N + (active ? (k * ny + j) * nx + x : 0);
    float2 wT = make_float2(0.f, 0.f);  // read ahead of its use: at its use it cost 30 us at 256^3
    if (t.w) wT = *reinterpret_cast<const float2*>(t.w + ready0 + oT);
    // Plane k + 2 takes the slot of plane k - 2, which every warp has read once it has done plane k - 1.  The first warp
    // alone waits for the others; they run on to the next plane by themselves.
    if (tid < 32 && k + 2 <= kend) {
      const int i = k - 1 - k0;
      if (i >= 0 && !__all_sync(0xffffffffu, bar_wait2(smem_addr2(&bar_done[i & 1]), (uint32_t)((i >> 1) & 1), err, spins)))
        ok = false;
      if (ok) {
        if (tid == 0) issue_plane(k + 2);
        issued = k + 2;
      }
    }
    ok = __all_sync(0xffffffffu, wait_plane(k + 1)) && ok;
    if (active && ok) {
      Ring2 S;
#pragma unroll
      for (int dz = -1; dz <= 1; ++dz)
        S.p[dz + 1] = sm + ((k + dz + kPRing) % kPRing) * kPNA * kPL2 + (ty + 1) * kPW2 + (2 * tx + kPX0);
      float2 conv, lap;
      const float2 msig = bc(-sigma);
      const int o = (k * ny + j) * nx + x;
      const float2 zero = make_float2(0.f, 0.f);
      {  // w: its low edges are u's and v's low z-edges
        const float2 aH = S.ld<2, 0, 0, 0>(), bH = S.ld<6, 0, 0, 0>(), bP = S.ld<6, 0, 0, 1>();
        const float2 half = bc(0.5f);
        const float2 fE = half * (aH + S.ld<2, 0, 0, 1>()) * (half * (bH + bP)), gE = (bP - bH) * mz.ix;
        conv = bc(2.f) * (fE - z.f[2]) * mz.ic;
        lap = (gE - z.g[2]) * mz.ic;
        z.f[2] = fE;
        z.g[2] = gE;
        across<2, 0>(S, mz, mx, aH, bH, z.f[0], conv, lap);
        across<2, 1>(S, mz, my, aH, bH, z.f[1], conv, lap);
        const float2 Tf = fma2(mz.wl, S.ld<7, 0, 0, -1>(), mz.wr * S.ld<7, 0, 0, 0>());
        const float2 r2 = fma2(msig, bH, fma2(bc(Gr), Tf, lap - conv));
        *reinterpret_cast<float2*>(out + 2 * N + o) = (k >= 1) ? r2 : zero;
      }
      float2 exy;  // the flux of the low x-y edge, u's and v's
      {
        const float2 aH = S.ld<0, 0, 0, 0>(), bH = S.ld<4, 0, 0, 0>();
        exy = edge_lo<0, 1>(S, mx, my, aH, bH, S.ld<4, 0, -1, 0>());
        along<0>(S, mx, aH, bH, conv, lap);
        across<0, 1>(S, mx, my, aH, bH, exy, conv, lap);
        across_z<0>(S, mx, mz, aH, bH, z.f[0], z.g[0], conv, lap);
        float2 r0 = fma2(msig, bH, lap - conv);
        if (x == 0) r0.x = 0.f;  // the x = 0 wall slot of u
        *reinterpret_cast<float2*>(out + o) = r0;
      }
      {
        const float2 aH = S.ld<1, 0, 0, 0>(), bH = S.ld<5, 0, 0, 0>();
        along<1>(S, my, aH, bH, conv, lap);
        across_z<1>(S, my, mz, aH, bH, z.f[1], z.g[1], conv, lap);
        across<1, 0>(S, my, mx, aH, bH, exy, conv, lap);
        const float2 r1 = fma2(msig, bH, lap - conv);
        *reinterpret_cast<float2*>(out + N + o) = (j >= 1) ? r1 : zero;
      }
      temperature_pair(S, mx, my, mz, j, ny, k, nz, z.f[3], z.g[3], conv, lap);
      const float2 r3 = fma2(msig, S.ld<7, 0, 0, 0>(), lap * bc(invPr) - conv);
      if (t.out) {
        float2 r = bc(t.alpha) * r3;
        if (t.add_v) r = fma2(bc(t.beta), S.ld<7, 0, 0, 0>(), r);
        if (t.w) r = fma2(bc(t.gamma), wT, r);
        *reinterpret_cast<float2*>(t.out + ready0 + oT) = r;
      } else {
        *reinterpret_cast<float2*>(out + 3 * N + o) = r3;
      }
    }
    __syncwarp();
    if ((tid & 31) == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr2(&bar_done[(k - k0) & 1])) : "memory");
  }
  // give-up path (a warp that stops arrives no more, so the first one runs into its limit too): every plane copy still in
  // flight lands (waited for with the full limit) before the CTA exits, so that no bulk copy writes into shared memory
  // the CTA no longer owns
  if (!ok && tid == 0)
    for (int kk = max(k0 - 1, issued - kPRing + 1); kk <= issued; ++kk)
      bar_wait2(smem_addr2(&bar[(kk + kPRing) % kPRing]), (uint32_t)(((kk - k0 + 1) / kPRing) & 1), err,
                kPWaitLimit);
}

// 4D tensor map of nvec FP32 states stored one after another (x, y, z, field; 4 nvec fields) with boxes
// of kPW2 x kPHY x 1 x 4 elements
int pair_map(const fv_grid_s* g, const float* ptr, CUtensorMap* m, int nvec = 1) {
  const uint64_t dims[4] = {(uint64_t)g->nx, (uint64_t)g->ny, (uint64_t)g->nz, 4 * (uint64_t)nvec};
  const uint64_t strides[3] = {g->nx * sizeof(float), (uint64_t)g->nx * g->ny * sizeof(float), g->N * sizeof(float)};
  const uint32_t box[4] = {(uint32_t)kPW2, (uint32_t)kPHY, 1, 4};
  return encode_tensor_map(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ptr, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}

}  // namespace

bool stencil_pair_eligible(const fv_grid_s* g, const float* q, const float* v) {
  return g->nx % kPX == 0 && g->ny >= 16 && ((uintptr_t)q % 16) == 0 && ((uintptr_t)v % 16) == 0;
}

int stencil_pair_setup() {
  for (auto k : {k_stencil_pair<false>, k_stencil_pair<true>})
    FV_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpreadSmem));
  return FV_OK;
}

int launch_stencil_pair(const fv_grid_s* g, double Gr, double sigma, const float* q, const float* v, float* out,
                        int nvec, const TempOut& t) {
  // blocks of vectors march the z-chunk the autotuner picked, if it ran; otherwise stencil_chunk's
  const int zc = (nvec > 1 && g->tune.pair_zc > 0) ? g->tune.pair_zc
                                                   : stencil_chunk(g->nz, g->sms, g->nx / kPX * ((g->ny + kPY - 1) / kPY), nvec, kPairTimes);
  const int nch = (g->nz + zc - 1) / zc;
  if (nvec < 1 || (long long)nch * nvec > 65535) {
    set_error("launch_stencil_pair: too many vectors in one block for this z-chunk");
    return FV_EINVAL;
  }
  CUtensorMap tq, tv;
  std::memset(&tq, 0, sizeof(tq));
  std::memset(&tv, 0, sizeof(tv));
  FV_TRY(pair_map(g, q, &tq));
  FV_TRY(pair_map(g, v, &tv, nvec));
  dim3 grid(g->nx / kPX, (g->ny + kPY - 1) / kPY, nch * nvec);
  const size_t smem = spread_smem(kPairSmem, (long long)grid.x * grid.y * grid.z, g->sms, kPairTimes.most);
  ProfScope ps(g, PROF_STENCIL);
  if (nvec > 1)
    launch(k_stencil_pair<true>, grid, kPX / 2 * kPY, smem, g->stream, tq, tv, g->ws.err, wait_spins(g), g->geo32, (int)g->N, (float)Gr,
                                                                 (float)(1.0 / g->Pr), (float)sigma, out, zc, nch, t);
  else
    launch(k_stencil_pair<false>, grid, kPX / 2 * kPY, smem, g->stream, tq, tv, g->ws.err, wait_spins(g), g->geo32, (int)g->N, (float)Gr,
                                                                  (float)(1.0 / g->Pr), (float)sigma, out, zc, nch, t);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

}  // namespace fv
