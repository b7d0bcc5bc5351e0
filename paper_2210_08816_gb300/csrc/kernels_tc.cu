// Fast-diagonalisation passes of the pressure solve for FP32 fields on the tensor cores (tcgen05), for grids whose axes
// have 32 .. 256 cells, a multiple of 32, and mirror-symmetric faces, stretched to s = 4 or so at most (tc_setup).
//
// A pass is the GEMM  C[p][m] = sum_k A[p][k] B[m][k]  (A = field rows, k contiguous; B = a 1D eigenvector matrix),
// stored transposed as out[m][p] (see kernels_fdm.cu), in the half-size form of HalfOpHost: forward passes contract
// the sums and differences of mirrored inputs with two h x h matrices (h = n / 2), backward passes write S +- A.
//
// FP32 accuracy on FP16 tensor cores: the field is scaled by one power of two into FP16's range (its largest
// magnitude below 2^14, found by the kernel that wrote it), and every sum or difference x is split as hi = fp16(x),
// lo = fp16(x - hi), 22 bits together; likewise the matrices (on the host, build_halves).  hi hi + hi lo + lo hi are
// accumulated in FP32; the dropped lo lo is 2^-24 of a product.  Values below 2^-17 of the field's largest keep an
// absolute error of 2^-39 of it.  Against the same three products of TF32 parts, which have the same mantissas: half
// the bytes per input in shared memory, half the MMA time, and half as many truncated accumulations (the projection's
// error against 64 bits falls from 0.83e-6 to 0.58e-6 at 64^3, from 2.0e-6 to 1.2e-6 at 256^3).
//
// One CTA per SM walks the 128-row tiles blockIdx.x, +gridDim.x, ... with all n outputs (rows and fields are whole
// tiles: a field has at least 32 x 32 rows).  Per step 32 inputs of each half: two TMA boxes of A (slab j and its mirror
// forward, slabs j and h + 32 j backward; 128-byte swizzle), the four B slabs (bulk copies of the pre-swizzled blocks;
// kept where all of B fits), and per k-step of 16 inputs 2 halves x 3 products of tcgen05.mma (M = 128, N = h, K = 16).
// Two TMEM accumulators (columns 0 and 256) let the epilogue of a tile run under the MMAs of the next.
// Warps: 0 TMA of A, 1 MMA issue, then converters, epilogue (8), bulk copies of B (the last).
// Barriers: afull / afree per raw stage (A landed / converted), bfull / bfree per B slab, conv / done per k-step
// (converted / MMAs complete); accf / acce per tile.  Every wait is bounded; on expiry the kernel records a code, stops
// issuing, lets its copies and MMAs complete and returns.
//
// What bounds it: the copies' arrival and the hand-offs of a step, not a unit.  256^3, six passes of 134 MB each: 198 us by
// themselves, ~150 within a time step's overlapping launches (TF32 parts: 222); DRAM 32 % (most of a field stays in L2
// between passes), L2 24 %.  Two stages of 32 KB of A arrive every ~1750 clocks per step.  More stages are slower (three:
// 630 us for the whole chebyshev step against 600), and so are equal row ranges instead of neighbouring tiles at a time
// (650): the writes are 512-byte pieces of n rows, and neighbours share DRAM pages.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <vector>

#include "fv_internal.h"
#include "launch.cuh"
#include "tcgen05.cuh"

namespace fv {
namespace {

constexpr int kTcBM = 128;                  // rows per tile
constexpr int kTcBK = 32;                   // inputs of a half per step: one 128-byte FP32 row, one 64-byte FP16 row
constexpr int kTcABytes = kTcBM * kTcBK * 4;  // one raw A slab (16 KB)
constexpr int kTcCBytes = kTcBM * kTcBK * 2;  // one converted slab (8 KB)
constexpr int kTcRing = 2;                    // raw stages
constexpr int kTcSteps = 4;  // converted k-steps of 16 inputs in flight, two to a slot of four slabs
constexpr int kTcEpi = 8;     // epilogue warps
constexpr size_t kTcSmemMost = 229376 + 1024;
constexpr int tc_threads(int conv) { return 64 + conv + 32 * kTcEpi + 32; }

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// approximate reciprocal (PTX rcp.approx, relative error about 2^-23): far below the error of the parts
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// eight values as FP16 heads and remainders
__device__ __forceinline__ void split8(const float (&x)[8], uint4& h, uint4& l) {
  uint32_t hw[4], lw[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __half2 hh = __floats2half2_rn(x[2 * i], x[2 * i + 1]);
    const float2 f = __half22float2(hh);
    const __half2 ll = __floats2half2_rn(x[2 * i] - f.x, x[2 * i + 1] - f.y);
    hw[i] = *reinterpret_cast<const uint32_t*>(&hh);
    lw[i] = *reinterpret_cast<const uint32_t*>(&ll);
  }
  h = make_uint4(hw[0], hw[1], hw[2], hw[3]);
  l = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}

// The exponent field of a field's largest magnitude (its bits in a slot), at least 32 (zero and tiny fields).
__device__ __forceinline__ int max_exponent(const unsigned* slot) { return max((int)(__ldcg(slot) >> 23), 32); }

// A warp's largest magnitude into a field's slot (fmaxf drops NaNs: one shows as a NaN in the next pass whatever the
// scale).
__device__ __forceinline__ void max_to(unsigned* slot, float top) {
  const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
  if (threadIdx.x % 32 == 0) atomicMax(slot, m);
}

struct TcArgs {
  const unsigned char* B;  // blocks [part][group of 64 outputs][slab]: 64 rows hi, 64 rows lo, of 64 bytes
  const int* bexp;         // exponent of every output pair
  float* out;
  const float *lx, *ly, *lz;  // scaled pass: eigenvalues
  const unsigned* max_in;     // slot of every vector: the bits of its largest input magnitude
  unsigned *max_out, *max_reset;  // the same for the output; a consumed slot to clear (either may be null)
  int P, Ptot, n, nb;
  int bslots;   // B slabs in shared memory: all of them, or a ring of two
  int* err;
  long long spins;
};

// CONV: converter threads, 256 or 512
template <bool SCALE, bool BWD, int CONV>
__global__ void __launch_bounds__(tc_threads(CONV), 1)
    k_pass_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ TcArgs t) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar_afull[kTcRing], bar_afree[kTcRing], bar_bfull[4], bar_bfree[2],
      bar_conv[kTcSteps], bar_done[kTcSteps],
      bar_accf[2], bar_acce[2], bar_drain;
  __shared__ uint32_t tmem_slot;
  __shared__ float lz_s[256], col_s[128];
  const int n = t.n, h = n / 2, P = t.P;
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t base = smem_u32(smem);
  const int bslots = t.bslots;
  constexpr uint32_t conv0 = kTcRing * 2u * kTcABytes, b0 = conv0 + (kTcSteps / 2) * 4u * kTcCBytes;
  const uint32_t b_bytes = (uint32_t)h * 64u;  // one B slab
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int nst = (h + kTcBK - 1) / kTcBK;
  const int ntiles = t.Ptot / kTcBM;
  const int my_tiles = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  pdl_begin();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kTcRing; ++s) {
      mbar_init(smem_u32(&bar_afull[s]), 1);
      mbar_init(smem_u32(&bar_afree[s]), 16);
    }
    for (int s = 0; s < 4; ++s) mbar_init(smem_u32(&bar_bfull[s]), 1);
    for (int s = 0; s < kTcSteps; ++s) {
      mbar_init(smem_u32(&bar_conv[s]), 8);
      mbar_init(smem_u32(&bar_done[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bar_accf[b]), 1);
      mbar_init(smem_u32(&bar_acce[b]), kTcEpi);
    }
    for (int b = 0; b < 2; ++b) mbar_init(smem_u32(&bar_bfree[b]), 1);
    mbar_init(smem_u32(&bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (SCALE)
    for (int m = threadIdx.x; m < n; m += tc_threads(CONV)) lz_s[m] = t.lz[m];
  for (int m = threadIdx.x; m < h; m += tc_threads(CONV)) col_s[m] = __int_as_float((t.bexp[m] + 127) << 23);
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  if (warp == 2 + CONV / 32 + kTcEpi) {
    // B, slab by slab as [half][hi | lo] of b_bytes each: kept for the CTA's lifetime where it fits, else around a ring
    // of two.  It is the grid's own, so the copies start before the kernel before this one has ended.
    if (lane == 0) {
      const int groups = (h + 63) / 64, loads = bslots == nst ? nst : my_tiles * nst;
      int issued = 0;
      for (; issued < loads; ++issued) {
        const int st = issued % bslots, j = issued % nst;
        if (issued >= bslots &&
            !mbar_wait(smem_u32(&bar_bfree[st]), ((issued / bslots) - 1) & 1, t.err, 13, t.spins))
          break;
        const uint32_t sb = base + b0 + st * 4u * b_bytes, fb = smem_u32(&bar_bfull[st]);
        mbar_expect_tx(fb, 4u * b_bytes);
        for (int part = 0; part < 2; ++part)
          for (int gr = 0; gr < groups; ++gr) {
            const uint32_t bytes = (uint32_t)std::min(64, h - 64 * gr) * 64u;
            const unsigned char* src = t.B + ((size_t)(part * groups + gr) * nst + j) * 8192;
            bulk_load(sb + (2 * part) * b_bytes + gr * 4096u, src, bytes, fb);
            bulk_load(sb + (2 * part + 1) * b_bytes + gr * 4096u, src + 4096, bytes, fb);
          }
      }
      // every issued copy has landed before the block may exit
      for (int i = std::max(issued - bslots, 0); i < issued; ++i)
        mbar_wait(smem_u32(&bar_bfull[i % bslots]), (i / bslots) & 1, t.err, 12, kWaitLimit);
    }
    __syncwarp();
  }
  // every role waits for the kernel before this one by itself, right where it first needs its results (the code up to
  // there has then been fetched; a wait of the whole block here cost 1 us of a pass in instruction misses)
  if (warp == 0) {
    if (lane == 0) {
      int gi = 0, issued = 0;
      bool ok = true;
      for (int ti = 0; ti < my_tiles && ok; ++ti) {
        const int p0 = ((int)blockIdx.x + ti * (int)gridDim.x) * kTcBM;
        for (int j = 0; j < nst; ++j, ++gi) {
          const int st = gi % kTcRing;
          if (gi >= kTcRing && !mbar_wait(smem_u32(&bar_afree[st]), ((gi / kTcRing) - 1) & 1, t.err, 11, t.spins)) {
            ok = false;
            break;
          }
          const uint32_t sa = base + st * 2u * kTcABytes, fb = smem_u32(&bar_afull[st]);
          const int x1 = j * kTcBK, x2 = BWD ? h + j * kTcBK : n - kTcBK - j * kTcBK;
          mbar_expect_tx(fb, 2u * kTcABytes);
          if (gi == 0) pdl_wait();
          tma_load_2d(sa, &tmA, fb, x1, p0);
          tma_load_2d(sa + kTcABytes, &tmA, fb, x2, p0);
          ++issued;
        }
      }
      // every issued copy has landed before the block may exit
      for (int g2 = std::max(issued - kTcRing, 0); g2 < issued; ++g2)
        mbar_wait(smem_u32(&bar_afull[g2 % kTcRing]), (g2 / kTcRing) & 1, t.err, 12, kWaitLimit);
    }
  } else if (warp == 1) {
    // descriptors differ from the first slab's by multiples of 16 bytes: additions only (building each from its
    // address in one lane cost 140 clocks per MMA, more than the MMA's own 64)
    const uint64_t desc0 = smem_desc(base);
    const uint32_t idesc = (1u << 4) | ((uint32_t)(h >> 3) << 17) | ((uint32_t)(kTcBM >> 4) << 24);
    int g2 = 0, gi = 0;  // k-steps of 16 inputs, steps of 32
    bool ok = true;
    for (int ti = 0; ti < my_tiles && ok; ++ti) {
      const int b = ti & 1;
      if (ti >= 2 &&
          !__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_acce[b]), ((ti / 2) - 1) & 1, t.err, 13, t.spins))) {
        ok = false;
        break;
      }
      const uint32_t dacc = tmem + (uint32_t)(b * 256);
      for (int j = 0; j < nst && ok; ++j, ++gi) {
        const int bs = gi % bslots;
        if ((ti == 0 || bslots < nst) &&
            !__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_bfull[bs]), (gi / bslots) & 1, t.err, 14, t.spins))) {
          ok = false;
          break;
        }
        const uint64_t db = desc0 + ((b0 + bs * 4u * b_bytes) >> 4);
        for (int kk = 0; kk < 2; ++kk, ++g2) {
          const int st = g2 % kTcSteps;
          if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_conv[st]), (g2 / kTcSteps) & 1, t.err, 15, t.spins))) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t dc = desc0 + ((conv0 + (st >> 1) * 4u * kTcCBytes + 32u * kk) >> 4);
          if (elect_one()) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              const uint64_t a_hi = dc + ((2u * half * kTcCBytes) >> 4), a_lo = a_hi + (kTcCBytes >> 4);
              const uint64_t b_hi = db + 2u * half * (uint64_t)(b_bytes >> 4) + 2 * kk, b_lo = b_hi + (b_bytes >> 4);
              const uint32_t d = dacc + (uint32_t)(half * h);
              mma_f16(d, a_hi, b_hi, idesc, (uint32_t)(j + kk > 0));
              mma_f16(d, a_hi, b_lo, idesc, 1u);
              mma_f16(d, a_lo, b_hi, idesc, 1u);
            }
            mma_commit(smem_u32(&bar_done[st]));
            if (kk == 1 && bslots < nst) mma_commit(smem_u32(&bar_bfree[bs]));
            if (kk == 1 && j == nst - 1) mma_commit(smem_u32(&bar_accf[b]));  // once every MMA so far has completed
          }
          __syncwarp();
        }
      }
    }
    // A commit after every MMA issued so far arrives once they have all completed; wait for it (full limit) before the
    // accumulators are freed and the block may exit, whoever gave up: the epilogue's wait for the last tiles can run out
    // when this warp has issued everything
    if (elect_one()) mma_commit(smem_u32(&bar_drain));
    mbar_wait(smem_u32(&bar_drain), 0, t.err, 16, kWaitLimit);
  } else if (warp < 2 + CONV / 32) {
    // converters: four threads to a row of every slab; those of one half of the warps take the first k-step of each
    // raw stage, the others the second, a thread inputs 8 hf .. 8 hf + 7 of it
    const int tt = threadIdx.x - 64, r = tt & 127, hf = (tt >> 7) & 1;
    const unsigned* max_in = t.max_in + pdl_wait();
    int gi = 0;
    bool ok = true;
    for (int ti = 0; ti < my_tiles && ok; ++ti) {
      const int vec = ((int)blockIdx.x + ti * (int)gridDim.x) * kTcBM / P;
      const float scale = __uint_as_float((unsigned)(267 - max_exponent(max_in + 8 * vec)) << 23);  // 2^(140 - E)
      for (int j = 0; j < nst && ok; ++j, ++gi) {
        const int st = gi % kTcRing;
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_afull[st]), (gi / kTcRing) & 1, t.err, 17, t.spins))) {
          ok = false;
          break;
        }
        for (int kk = tt >> 8; kk < 2 && ok; kk += CONV / 256) {
          const int g2 = 2 * gi + kk, sk = g2 % kTcSteps;
          uint4 sh, sl, dh, dl;
          const unsigned char* raw = smem + st * 2u * kTcABytes + r * 128;
          float s[8], d[8];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int ca = 4 * kk + 2 * hf + c, cm = BWD ? ca : 7 - ca;  // forward: the mirrors in reverse order
            const float4 x = *reinterpret_cast<const float4*>(raw + ((ca ^ (r & 7)) << 4));
            const float4 y = *reinterpret_cast<const float4*>(raw + kTcABytes + ((cm ^ (r & 7)) << 4));
            const float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float m = BWD ? ys[e] : ys[3 - e];
              s[4 * c + e] = (BWD ? xs[e] : xs[e] + m) * scale;
              d[4 * c + e] = (BWD ? m : xs[e] - m) * scale;
            }
          }
          split8(s, sh, sl);
          split8(d, dh, dl);
          // the k-step's part of the slot was last read by the MMAs of k-step g2 - kTcSteps
          if (g2 >= kTcSteps &&
              !__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_done[sk]), ((g2 / kTcSteps) - 1) & 1, t.err, 19, t.spins))) {
            ok = false;
            break;
          }
          unsigned char* dst =
              smem + conv0 + (sk >> 1) * 4u * kTcCBytes + r * 64 + (((2 * kk + hf) ^ ((r >> 1) & 3)) << 4);
          *reinterpret_cast<uint4*>(dst) = sh;
          *reinterpret_cast<uint4*>(dst + kTcCBytes) = sl;
          *reinterpret_cast<uint4*>(dst + 2 * kTcCBytes) = dh;
          *reinterpret_cast<uint4*>(dst + 3 * kTcCBytes) = dl;
          // the fence also stands between this thread's reads of the raw stage and its release: an arrival directly
          // after the loads let the next copy overtake them
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(smem_u32(&bar_conv[sk]));
            mbar_arrive(smem_u32(&bar_afree[st]));
          }
        }
      }
    }
  } else if (warp < 2 + CONV / 32 + kTcEpi) {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31, one row of the tile per thread; the two warps of a quadrant
    // take alternate chunks of 16 outputs
    const int row = (warp % 4) * 32 + lane, half = (warp - 2 - CONV / 32) / 4;
    const unsigned ready0 = pdl_wait();
    const unsigned* max_in = t.max_in + ready0;
    if (blockIdx.x == 0)  // a slot that the kernel before this one has read
      for (int v = threadIdx.x - 64 - CONV; v * P < t.Ptot; v += 32 * kTcEpi) t.max_reset[8 * v] = 0;
    float top = 0.f;  // the largest output of field top_vec so far
    int top_vec = 0;
    for (int ti = 0; ti < my_tiles; ++ti) {
      const int b = ti & 1;
      // row p of field vec (fields of P x n, one after another)
      const int p0 = ((int)blockIdx.x + ti * (int)gridDim.x) * kTcBM, vec = p0 / P, p = p0 + row - vec * P;
      float* __restrict__ o = t.out + ready0 + (size_t)vec * P * n + p;
      float sa = 0.f, sb = 0.f;
      bool null_row = false;
      if (SCALE) {
        const int pa = p / t.nb;
        sa = t.ly[pa];
        sb = t.lx[p - pa * t.nb];
        null_row = p == 0;
      }
      // 2^(E - 140); a field with an Inf or NaN keeps them through the splits
      const float row_scale = __uint_as_float((unsigned)(std::min(max_exponent(max_in + 8 * vec), 254) - 13) << 23);
      const bool ok = mbar_wait(smem_u32(&bar_accf[b]), (ti / 2) & 1, t.err, 18, t.spins);
      if (!__all_sync(0xffffffffu, ok)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t lane_base = tmem + ((uint32_t)((warp % 4) * 32) << 16) + (uint32_t)(b * 256);
      if (t.max_out && vec != top_vec) {
        if (ti > 0) max_to(t.max_out + 8 * top_vec, top);
        top = 0.f;
        top_vec = vec;
      }
      for (int c0 = 16 * half; c0 < h; c0 += 32) {
        uint32_t r1[16], r2[16];
        tmem_ld16(lane_base + (uint32_t)c0, r1);
        tmem_ld16(lane_base + (uint32_t)(h + c0), r2);
        float* __restrict__ o1 = o + (size_t)c0 * P;
        float* __restrict__ o2 = o + (size_t)(BWD ? n - 1 - c0 : h + c0) * P;
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) {
          const float cs = col_s[c0 + jj];
          float v1 = __uint_as_float(r1[jj]) * cs, v2 = __uint_as_float(r2[jj]) * cs;
          if (BWD) {  // cells m and n-1-m
            const float s = v1 + v2;
            v2 = v1 - v2;
            v1 = s;
          }
          v1 *= row_scale;
          v2 *= row_scale;
          if (SCALE) {  // symmetric mode m, antisymmetric mode h + m
            const int m = c0 + jj;
            v1 = (m == 0 && null_row) ? 0.f : v1 * rcp_approx(lz_s[m] + sa + sb);
            v2 *= rcp_approx(lz_s[h + m] + sa + sb);
          }
          top = fmaxf(top, fmaxf(fabsf(v1), fabsf(v2)));
          *o1 = v1;
          *o2 = v2;
          o1 += P;
          o2 += BWD ? -P : P;
        }
      }
      // the accumulator's values are in registers (tcgen05.wait::ld): the MMAs may reuse it
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_acce[b]));
    }
    if (t.max_out) max_to(t.max_out + 8 * top_vec, top);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encoder() {
  static EncodeFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  }
  return fn;
}

// rows x cols FP32 row-major matrix (cols contiguous), boxes of 32 columns x 128 rows, 128-byte swizzle
int encode(CUtensorMap* m, const float* ptr, long long rows, int cols) {
  const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows};
  const uint64_t strides[1] = {(uint64_t)cols * 4};
  const uint32_t box[2] = {(uint32_t)kTcBK, (uint32_t)kTcBM};
  return encode_tensor_map(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, ptr, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

// Shared memory of a pass of n outputs: the raw stages, the converted slots and B, all of it where it fits, else a ring
// of two slabs.
size_t tc_layout(int n, int& bslots) {
  const int h = n / 2, nst = (h + kTcBK - 1) / kTcBK;
  const size_t fixed = kTcRing * 2 * kTcABytes + (kTcSteps / 2) * 4 * kTcCBytes + 1024, slab = (size_t)4 * h * 64;
  bslots = fixed + nst * slab <= kTcSmemMost ? nst : 2;
  return fixed + bslots * slab;
}

}  // namespace

int encode_tensor_map(CUtensorMap* map, CUtensorMapDataType type, int rank, const void* ptr, const uint64_t* dims,
                      const uint64_t* strides, const uint32_t* box, CUtensorMapSwizzle swizzle) {
  EncodeFn fn = encoder();
  if (!fn) {
    set_error("cuTensorMapEncodeTiled unavailable");
    return FV_ECUDA;
  }
  cuuint64_t d[5], st[4];
  cuuint32_t b[5], e[5];
  for (int i = 0; i < rank; ++i) {
    d[i] = dims[i];
    b[i] = box[i];
    e[i] = 1;
    if (i + 1 < rank) st[i] = strides[i];
  }
  const CUresult r = fn(map, type, (cuuint32_t)rank, const_cast<void*>(ptr), d, st, b, e, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed");
    return FV_ECUDA;
  }
  return FV_OK;
}

// The grid's FP32 pressure solves take these passes (half-size operators and their FP16 parts are ready).
// Not on strongly stretched grids: the parts keep 2^-39 of the field's largest value, and a corner cell's potential is put
// together from coefficients smaller than that value by the square root of the product of the axes' width ratios.  Up to a
// product of 2^29 what is lost stays below FP32's own rounding (2^-24); beyond it the passes with a scale per row
// (kernels_digit.cu) or FP32 sums take over.  Projection's error, 128 x 64 x 32, s = 2, 3, 4, 6 (products 2^11, 2^20, 2^28,
// 2^45): here 1.3e-6, 4.9e-6, 3.0e-5, 4.8e-2; FP32 sums of TF32 parts 1.7e-6, 5.4e-6, 3.5e-5, 1.3e-3; with a scale per row
// 5e-7, 2e-6, 1.4e-5, 7e-4 (130 x 70 x 60).  Time of a 256^3 projection 337 us here, 593 with a scale per row.
constexpr double kTcMostSpan = 536870912.0;
int tc_setup(fv_grid_s* g) {
  static_assert(kDigitCols32 == 64 && kDigits32 == 2, "the B blocks hold 64 outputs, two parts");
  const int n[3] = {g->nx, g->ny, g->nz};
  if (!tc_sizes(n)) return FV_OK;
  if (width_ratio(g->xf[0]) * width_ratio(g->xf[1]) * width_ratio(g->xf[2]) > kTcMostSpan) return FV_OK;
  if (!g->digit_ready || !encoder()) return FV_OK;
  for (auto k : {k_pass_tc<false, false, 256>, k_pass_tc<true, false, 256>, k_pass_tc<false, true, 256>,
                 k_pass_tc<false, false, 512>, k_pass_tc<true, false, 512>, k_pass_tc<false, true, 512>})
    FV_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmemMost));
  g->tc_ready = true;
  return FV_OK;
}

// Pass 0 .. 5 of a solve (forward x, y, z, backward x, y, z): in[a][b][k] (na*nb rows of n) -> out[m][a][b].  Mode
// indices are in the half order throughout.  nvec > 1: that many fields of na*nb*n elements one after another in `in`
// and in `out`, each transformed alone, all in one launch.  slots: 8 words per field; pass i reads the field's largest
// magnitude in word i, leaves its output's in word i + 1 (not the last pass) and clears word i - 1 (the first pass:
// word 5), so that every word is zero again before the next solve writes it.
int tc_pass(const fv_grid_s* g, int pass, int na, int nb, const float* in, float* out, unsigned* slots, int nvec) {
  const int axis = pass % 3;
  const bool bwd = pass >= 3;
  const int n = (axis == 0) ? g->nx : (axis == 1) ? g->ny : g->nz;
  const long long P = (long long)na * nb, Ptot = P * nvec;
  if (nvec < 1 || Ptot > (1LL << 30)) {
    set_error("tc_pass: batch of fields not supported here");
    return FV_EINVAL;
  }
  CUtensorMap tmA;
  FV_TRY(encode(&tmA, in, Ptot, n));
  const HalfDev<float>& d = g->half32[axis][HALF_NEUMANN];
  TcArgs t{};
  t.B = d.dig[bwd ? 1 : 0];
  t.bexp = d.dexp[bwd ? 1 : 0];
  t.out = out;
  t.lx = g->half32[0][HALF_NEUMANN].lam;
  t.ly = g->half32[1][HALF_NEUMANN].lam;
  t.lz = g->half32[2][HALF_NEUMANN].lam;
  t.max_in = slots + pass;
  t.max_out = pass < 5 ? slots + pass + 1 : nullptr;
  t.max_reset = slots + (pass + 5) % 6;
  t.P = (int)P;
  t.Ptot = (int)Ptot;
  t.n = n;
  t.nb = nb;
  const size_t smem = tc_layout(n, t.bslots);
  t.err = g->ws.err;
  t.spins = wait_spins(g);
  const long long ntiles = Ptot / kTcBM;
  const dim3 grid((unsigned)std::min<long long>(ntiles, g->sms));
  ProfScope ps(g, PROF_TRANSFORM_TC);
  // twice the converters from five steps a tile on (256^3 chebyshev step 613 -> 602 us); with fewer steps the larger
  // block's start costs more than they save (64^3 product 47 -> 49 us)
  auto go = [&](auto conv) {
    constexpr int C = decltype(conv)::value;
    auto k = bwd ? k_pass_tc<false, true, C> : pass == 2 ? k_pass_tc<true, false, C> : k_pass_tc<false, false, C>;
    launch(k, grid, tc_threads(C), smem, g->stream, tmA, t);
  };
  if (n > 128)
    go(std::integral_constant<int, 512>());
  else
    go(std::integral_constant<int, 256>());
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

}  // namespace fv
