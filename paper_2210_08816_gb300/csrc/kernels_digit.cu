// Fast-diagonalisation passes on the tensor cores by products of FP16 parts (tcgen05.mma kind::f16): FP64 fields, and
// FP32 fields of any size and operator.
//
// A pass contracts the sums and differences of mirrored inputs with two h x h matrices (see HalfOpHost).
//
// FP64: exact digit products, the error-free splitting of Ozaki, Ogita, Oishi & Rump (Numer. Algorithms 59, 2012) with
// fixed-point rows.  Each row of inputs is written on a common exponent as an integer of 7 balanced base-256 digits,
// x = 2^e sum_i x_i 256^(6-i), |x_i| <= 128, and so is each row of a matrix (on the host, build_digits).  Digits are
// exact in FP16, a product of two is at most 2^14, and the sum over K <= 128 inputs of the at most 7 products of one
// order i + j is an integer of at most 2^24: FP32 accumulators hold it exactly.  Orders 0 .. 6 are kept (28 products;
// the first dropped one lies 2^-56 below the row's largest product) and joined in the epilogue as a 64-bit integer,
// so the only roundings are the digits' quantisation, the dropped orders and the conversion of the result.
// These are absolute in a row, so what a row spans must not be spanned by its inputs and its matrix separately.  The
// matrices of a stretched axis do: the modes of the narrow cells have entries larger than the others' by the square root of
// the ratio of the widths, and coefficients as much smaller.  Every column is therefore brought into the same binade on the
// host and its inputs are lowered by as much (cexp: an integer addition to their exponents).
//
// FP32: rows scaled by a power of two into FP16's range, every value as the sum of two FP16 numbers (23 bits), all four
// products, with the leading one spread over two accumulators.  (Fixed-point digits as in FP64 would need 32 bits: with
// 25 their error, absolute in a row, was up to 4 times that of FP32 arithmetic on stretched grids.)
//
// Why: GB300 issues two FP64 operations per clock and SM (1.23 TFLOP/s measured in k_half); the 28 FP16 products
// cost 155 GFLOP per 256^3 pass where the FP16 tensor rate is 1.9 PFLOP/s.  Measured, six passes, CUDA cores / here:
// FP64 256^3 21.9 / 2.00 ms, 100^3 794 / 199 us; FP32 100^3 88 / 75 us, 250^3 1360 / 460 us, four fields of 256^3
// 5.2 / 1.67 ms.  Errors against 64 bits are at or below those of the CUDA-core passes (FP32 100^3 product 3.9e-7 ->
// 2.4e-7, FP64 256^3 3.4e-14 as before).  What bounds a unit is the workers' instruction issue (FP64: digits and the
// joining of the accumulators, 56 % of the integer pipe), not the MMAs (19 % of the tensor pipe).
//
// Layout (FP64).  Stacking the matrix digits j = 0 .. D-1-i of NC outputs as rows of one B operand makes all products of
// input digit i ONE instruction: N = (D - i) NC columns, accumulated at column i NC, where block d of NC columns
// holds order d.  (FP32: blocks hi hi twice, then the rest.)  A unit of work is 128, 96 or 32 rows x NC pairs, both
// parts; TMEM columns 0 and 256 hold the symmetric and the antisymmetric accumulators.  A CTA walks a contiguous range
// of units (the groups of NC pairs of a tile follow
// each other, so its rows stay in L2 and their exponents are found once).  Warps:
//   0      bulk copies of the B digits (pre-swizzled blocks) into the slots of a ring
//   1      TMEM allocation, MMA issue
//   2-17   workers: row exponents, then per slab of 32 inputs the sum and difference digits into two slots; the
//          epilogue of unit u (four warps per TMEM lane quadrant) between the first and the second slab of unit
//          u + 1, so that the MMAs find digits waiting when the accumulators are free
// Barriers per slot: full (B landed), conv (all workers), empty (commit); per unit accf (commit) and acce.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "fv_internal.h"
#include "launch.cuh"
#include "tcgen05.cuh"

namespace fv {
namespace {

constexpr int kDgRows = 128;
constexpr int kDgWarps = 16;  // workers
constexpr int kDgThreads = 32 * (2 + kDgWarps);
constexpr int kDgDigitBytes = kDgRows * 64;  // one digit of a 128 x 32 slab (64-byte swizzled rows)

// D digits per value, NC outputs per unit, ACC accumulators per output, E outputs of a row read from TMEM at a time,
// slots of the ring; the type a scaled input has and the type the joined accumulators have
template <typename R>
struct Dg;
template <>
struct Dg<double> {
  static constexpr int D = kDigits64, NC = kDigitCols64, ACC = D, E = 2, kSlots = 3;
  using Val = long long;
};
template <>
struct Dg<float> {
  static constexpr int D = kDigits32, NC = kDigitCols32, ACC = 3, E = 4, kSlots = 6;
  using Val = float;
};

template <typename R>
struct DgArgs {
  const unsigned char* B[4];  // per operator: digit blocks [part][group][slab] of this direction
  const int* eM[4];           // per operator: exponent of every output pair
  const unsigned char* cM[4];  // FP64, per operator: what the exponents of a column's inputs are lowered by
  const R* lam[3][4];         // scaled pass: eigenvalues of the three axes per operator
  R fac[4], shift[4];         // scaled pass: fac / (lam_z + lam_y + lam_x - shift)
  int k0[4], S[4];
  int P, n, nb, op_mask, scale, zero_mode;
  int tiles, groups, nslab, units, vec;
  int* err;
  long long spins;
};

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[2]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

__device__ __forceinline__ unsigned magnitude_bits(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned magnitude_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }

// x on the row's exponent E.  FP64: an integer, truncated, |I| < 2^54 with value I 2^(E - 1076); E >= 64 and shifts
// clamp, so that zeros and subnormals shift out (the dropped bits lie below 2^-53 of the row's largest input, a
// fraction of what the roundings of an FMA chain over its inputs add up to).  x 2^-c: E + c instead of E.  FP32: scaled
// below 2^14, value y 2^(E - 140).
__device__ __forceinline__ long long scaled(double x, int E) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  unsigned long long m = (((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32) | lo) << 1;
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(E - (int)(((unsigned)hi & 0x7fffffffu) >> 20)));
  const long long sg = (long long)(hi >> 31);
  return ((long long)m ^ sg) - sg;
}
__device__ __forceinline__ float scaled(float x, int E) { return x * __uint_as_float((unsigned)(267 - E) << 23); }

// The high word of |x| 2^-c (0 where it would fall below the smallest exponent; an Inf or NaN keeps its own)
__device__ __forceinline__ unsigned lowered(unsigned high, int c) {
  return high >= 0x7ff00000u ? high : (unsigned)max((int)high - (c << 20), 0);
}

// The D digits of two neighbouring inputs as FP16 pairs, digit i at dst + i * kDgDigitBytes.  FP64: balanced base-256
// digits; adding 128 to each makes them the bytes of an unsigned integer; 0x6400 | byte is the FP16 number
// 1024 + byte.
__device__ __forceinline__ void put_pair(unsigned char* dst, uint32_t h) {
  const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(0xE480)));  // - 1152
  *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(&r);
}
// digits lo and lo - 1 of both inputs from the low (sel 0x5410) or high (0x7632) halves of their words
__device__ __forceinline__ void put_two(unsigned char* dst, int lo, uint32_t a, uint32_t b, uint32_t sel) {
  const uint32_t w = __byte_perm(a, b, sel);
  put_pair(dst + lo * kDgDigitBytes, __byte_perm(w, 0x64646464u, 0x4240));
  put_pair(dst + (lo - 1) * kDgDigitBytes, __byte_perm(w, 0x64646464u, 0x4341));
}
__device__ __forceinline__ void put_digits(unsigned char* dst, long long I0, long long I1) {
  constexpr unsigned long long kBias = 0x80808080808080ull;
  const unsigned long long u0 = (unsigned long long)I0 + kBias, u1 = (unsigned long long)I1 + kBias;
  const uint32_t a0 = (uint32_t)u0, a1 = (uint32_t)(u0 >> 32), b0 = (uint32_t)u1, b1 = (uint32_t)(u1 >> 32);
  put_two(dst, 6, a0, b0, 0x5410);
  put_two(dst, 4, a0, b0, 0x7632);
  put_two(dst, 2, a1, b1, 0x5410);
  put_pair(dst, __byte_perm(a1, b1, 0x7632) | 0x64006400u);  // the leading digit may be 256 - 128
}
// FP32: the value rounded to FP16 and the remainder rounded to FP16
__device__ __forceinline__ void put_digits(unsigned char* dst, float y0, float y1) {
  const __half2 h = __floats2half2_rn(y0, y1);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(y0 - f.x, y1 - f.y);
  *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(&h);
  *reinterpret_cast<uint32_t*>(dst + kDgDigitBytes) = *reinterpret_cast<const uint32_t*>(&l);
}

// Inputs: FP32 passes by plain expressions, FP64 ones by loads that may pass stores (256^3 FP32 diffusion solve 1642 and
// 1666 us, 100^3 FP64 513 and 507).
template <typename R, typename T>
__device__ __forceinline__ T load_in(const T* p) {
  if constexpr (sizeof(R) == 8)
    return load_global(p);
  else
    return *p;
}

// Two neighbouring values: one vector load when `vec` (the pair is aligned), else two scalar ones; the second only
// if `two`.
template <typename R>
__device__ __forceinline__ void load_two(const R* p, bool vec, bool two, R& a, R& b) {
  if (vec) {
    using V2 = typename std::conditional<sizeof(R) == 8, double2, float2>::type;
    const V2 v = load_in<R>(reinterpret_cast<const V2*>(p));
    a = v.x;
    b = v.y;
  } else {
    a = load_in<R>(p);
    b = two ? load_in<R>(p + 1) : R(0);
  }
}

// The D order sums of one output joined.  FP64: an integer V = 2^-8 sum_d A_d 256^(6-d) (value V 2^(E + eM -
// 1020)), |V| < 2^62 so that S +- A fits.
__device__ __forceinline__ long long join_orders(const uint32_t (&r)[7][2], int j) {
  auto A = [&](int d) { return __float2int_rn(__uint_as_float(r[d][j])); };
  const long long hi = (long long)(A(1) * 256 + A(2)) * 16777216 + ((long long)A(0) << 40);
  return hi + (long long)A(3) * 65536 + (long long)A(4) * 256 + (A(5) + (A(6) >> 8));
}
// FP32: the sum of all (value V 2^(E + eM - 140))
__device__ __forceinline__ float join_orders(const uint32_t (&r)[3][4], int j) {
  return (__uint_as_float(r[0][j]) + __uint_as_float(r[1][j])) + __uint_as_float(r[2][j]);
}

// v 2^e rounded to nearest; integer arithmetic only (an FP64 operation per output would cost as much as the MMAs).
// fast: |e| is small enough that the result is normal whatever v is (or zero).
__device__ __forceinline__ double from_fixed(long long v, int e, bool fast) {
  const long long sg = v >> 63;
  unsigned long long u = (unsigned long long)((v ^ sg) - sg);  // <= 2^62
  if (u == 0) return 0.0;
  const int lz = __clzll((long long)u) - 1;
  u = ((u << lz) + 512) >> 10;          // 53 bits, the leading one at bit 52 (or 53 after rounding up)
  const int be = e + 62 - lz + 1023;    // biased exponent
  unsigned long long b = u + ((unsigned long long)(unsigned)(be - 1) << 52);
  if (!fast) b = be >= 2047 ? 0x7ff0000000000000ull : be < 1 ? 0ull : b;
  return __longlong_as_double((long long)(b | ((unsigned long long)sg << 63)));
}
template <typename R>
__device__ __forceinline__ R quiet_nan();
template <>
__device__ __forceinline__ double quiet_nan<double>() { return __longlong_as_double(0x7ff8000000000000LL); }
template <>
__device__ __forceinline__ float quiet_nan<float>() { return __uint_as_float(0x7fc00000u); }

// A unit of work (field, tile of rows, group of outputs), stepped without divisions: every warp keeps its own, and
// the integer divisions of a fresh decomposition per slab cost the workers as much as a slab's conversion.
template <typename R>
struct DgUnit {
  int group, tile, field;
  __device__ __forceinline__ DgUnit(const DgArgs<R>& t, int u) {
    const int ft = u / t.groups;
    group = u - ft * t.groups;
    field = ft / t.tiles;
    tile = ft - field * t.tiles;
  }
  __device__ __forceinline__ void step(const DgArgs<R>& t) {
    if (++group == t.groups) {
      group = 0;
      if (++tile == t.tiles) tile = 0, ++field;
    }
  }
};

// ITS: row pairs of a worker warp per slab; tiles of kRowsT = 32 ITS rows (the MMAs take 128, what the others hold is
// not read)
template <typename R, bool BWD, int ITS>
__global__ void __launch_bounds__(kDgThreads, 1)
    k_digit_pass(const __grid_constant__ DgArgs<R> t, const R* in, R* __restrict__ out) {
  constexpr int kRowsT = 2 * kDgWarps * ITS;
  constexpr int D = Dg<R>::D, NC = Dg<R>::NC, ACC = Dg<R>::ACC, E_ = Dg<R>::E, kSlots = Dg<R>::kSlots;
  constexpr bool F64 = sizeof(R) == 8;
  constexpr int kExpShift = F64 ? 20 : 23, kExpMax = F64 ? 2047 : 255, kExpMin = F64 ? 64 : 32;
  constexpr uint32_t kABytes = D * kDgDigitBytes, kBBytes = D * NC * 64, kSlotBytes = kABytes + kBBytes;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[kSlots], bar_conv[kSlots], bar_empty[kSlots];
  __shared__ __align__(8) uint64_t bar_accf, bar_acce, bar_drain;
  __shared__ uint32_t tmem_slot;
  // exponents of the rows, four tiles deep: a warp can find those of tile T + 1 while another still reads T - 1's in
  // an epilogue (tile T + 2 has to wait for that epilogue's MMAs)
  __shared__ int row_exp[4][kDgRows];
  __shared__ unsigned char in_exp[4][2 * kDigitMaxH + 4];  // FP64: cM of every input of a row
  __shared__ int out_exp[4][kDigitMaxH];  // exponents of the matrix rows per operator (FP32: 2^exponent, as bits)
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t base = smem_u32(smem);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int n = t.n, P = t.P, h = (n + 1) / 2, ha = n / 2;
  pdl_begin();
  const int u0 = (int)((long long)t.units * blockIdx.x / gridDim.x);
  const int u1 = (int)((long long)t.units * (blockIdx.x + 1) / gridDim.x);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_conv[s]), 32 * kDgWarps);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    mbar_init(smem_u32(&bar_accf), 1);
    mbar_init(smem_u32(&bar_acce), kDgWarps);
    mbar_init(smem_u32(&bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < (t.op_mask + 1) * h; i += kDgThreads) 
    out_exp[i / h][i % h] = F64 ? t.eM[i / h][i % h] : (t.eM[i / h][i % h] + 127) << 23;  // FP32: the power of two
  if (F64)
    for (int i = threadIdx.x; i < (t.op_mask + 1) * n; i += kDgThreads) {
      const int op = i / n, r = i - op * n, k = r - t.k0[op];  // (forward: the cell k0 + k or its mirror)
      in_exp[op][r] = t.cM[op][BWD ? r : max(min(k, t.S[op] - t.k0[op] - r), 0)];
    }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  const unsigned ready0 = pdl_wait();
  in += ready0;
  out += ready0;

  if (warp == 0) {
    if (lane == 0) {
      int gi = 0, issued = 0;
      bool ok = true;
      DgUnit<R> un(t, u0), nx = un;
      for (int u = u0; u < u1 && ok; ++u) {
        const int group = un.group, op = un.field & t.op_mask;
        // the rows of the next tile into L2, while this one is worked on
        if (u == u0 || group == 0) {
          int v = u;
          do nx.step(t), ++v;
          while (nx.group != 0);
          if (v < u1) {
            const R* src = in + ((size_t)nx.field * P + (size_t)nx.tile * kRowsT) * n;
            const uint32_t bytes = (uint32_t)(min(kRowsT, P - nx.tile * kRowsT) * n * sizeof(R)) & ~15u;
            if ((uintptr_t)src % 16 == 0 && bytes)
              asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
          }
        }
        for (int j = 0; j < t.nslab && ok; ++j)
          for (int part = 0; part < 2; ++part, ++gi) {
            const int st = gi % kSlots;
            if (gi >= kSlots &&
                !mbar_wait(smem_u32(&bar_empty[st]), ((gi / kSlots) - 1) & 1, t.err, 31, t.spins)) {
              ok = false;
              break;
            }
            const uint32_t fb = smem_u32(&bar_full[st]);
            mbar_expect_tx(fb, kBBytes);
            bulk_load(base + st * kSlotBytes + kABytes,
                      t.B[op] + ((size_t)(part * t.groups + group) * t.nslab + j) * kBBytes, kBBytes, fb);
            ++issued;
          }
        un.step(t);
      }
      // every issued copy has landed before the block may exit
      for (int g2 = (issued > kSlots ? issued - kSlots : 0); g2 < issued; ++g2)
        mbar_wait(smem_u32(&bar_full[g2 % kSlots]), (g2 / kSlots) & 1, t.err, 32, kWaitLimit);
    }
  } else if (warp == 1) {
    // descriptors differ from the first slot's by constants: one addition per MMA (building each from its address in
    // one lane cost 140 clocks per MMA, more than the MMA itself: 64 on average)
    const uint64_t desc0 = smem_desc(base);
    int gi = 0;
    bool ok = true;
    for (int u = u0; u < u1 && ok; ++u) {
      if (u > u0 && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_acce), (u - u0 - 1) & 1, t.err, 33, t.spins))) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int j = 0; j < t.nslab && ok; ++j)
        for (int part = 0; part < 2; ++part, ++gi) {
          const int st = gi % kSlots;
          const uint32_t ph = (gi / kSlots) & 1;
          if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_full[st]), ph, t.err, 34, t.spins) &&
                                           mbar_wait(smem_u32(&bar_conv[st]), ph, t.err, 35, t.spins))) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = desc0 + (uint64_t)((st * kSlotBytes) >> 4), db = da + (kABytes >> 4);
          const uint32_t acc = tmem + part * 256;
          if (elect_one()) {
            // M = 128, FP16 operands, FP32 accumulators
            auto mma = [&](int col, int i, int row, int cols, int kk, bool acc_on) {  // input digit i, B rows from `row`
              constexpr uint32_t kId = (1u << 4) | ((kDgRows / 16u) << 24);
              mma_f16(acc + col, da + ((i * kDgDigitBytes + kk * 32) >> 4), db + ((row * 64 + kk * 32) >> 4),
                      kId | ((uint32_t)(cols / 8) << 17), acc_on ? 1u : (uint32_t)(j > 0));
            };
            if constexpr (F64) {
#pragma unroll
              for (int kk = 0; kk < 2; ++kk)
#pragma unroll
                for (int i = 0; i < D; ++i) mma(i * NC, i, 0, (D - i) * NC, kk, kk > 0 || i > 0);
            } else {
              // hi hi into two accumulators by turns (the tensor cores truncate their sums: half the steps, half the
              // bias), the cross products and lo lo into the third
              mma(0, 0, 0, NC, 0, false);
              mma(2 * NC, 0, NC, NC, 0, false);
              mma(2 * NC, 1, 0, NC, 0, true);
              mma(2 * NC, 1, NC, NC, 0, true);
              mma(NC, 0, 0, NC, 1, false);
              mma(2 * NC, 0, NC, NC, 1, true);
              mma(2 * NC, 1, 0, NC, 1, true);
              mma(2 * NC, 1, NC, NC, 1, true);
            }
            mma_commit(smem_u32(&bar_empty[st]));
            // (the last slab's second part: arrives once every MMA of the unit has completed)
            if (part == 1 && j == t.nslab - 1) mma_commit(smem_u32(&bar_accf));
          }
          __syncwarp();
        }
    }
    // Whoever gives up (a worker's wait for the last unit can run out when this warp has issued everything): wait (full
    // limit) for every MMA issued so far before the accumulators are freed and the block may exit
    if (elect_one()) mma_commit(smem_u32(&bar_drain));
    mbar_wait(smem_u32(&bar_drain), 0, t.err, 36, kWaitLimit);
  } else {
    // a worker warp converts rows 2 (kDgWarps it + cw), + 1 (half a warp each; a lane takes two neighbouring input
    // pairs) and reads TMEM lanes 32 (warp % 4) .. + 31 in the epilogue (one row per thread)
    const int cw = warp - 2, rh = lane >> 4, kl = (lane & 15) * 2;
    const bool vec = t.vec != 0;
    const int erow = (warp % 4) * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)((warp % 4) * 32) << 16);
    const int total = (u1 - u0) * t.nslab;
    int item = 0, tc = 0;  // slabs done; count of tiles (row_exp)
    bool ok = true;
    DgUnit<R> un(t, u0), nx = un, pv = un;  // this unit, the next slab's, the one before
    // inputs of row pair `it` for the slab of an item; those of the next slab are requested as soon as this one's
    // are converted
    R x0[ITS], x1[ITS], y0[ITS], y1[ITS];
    auto load_row = [&](int it, const R* src, int rows, int k, int k0, int S) {
      const int row = 2 * (kDgWarps * it + cw) + rh;
      const bool two = k + 1 < h;
      x0[it] = x1[it] = y0[it] = y1[it] = R(0);
      if (k < h && row < rows) {
        const R* p = src + (size_t)row * n;
        if (BWD) {
          load_two<R>(p + k, vec, two, x0[it], x1[it]);
          if (k < ha) load_two<R>(p + h + k, vec, k + 1 < ha, y0[it], y1[it]);
        } else if (vec && two) {
          load_two<R>(p + k0 + k, true, true, x0[it], x1[it]);
          load_two<R>(p + S - k0 - k - 1, true, true, y1[it], y0[it]);
        } else {
          load_two<R>(p + k0 + k, false, two, x0[it], x1[it]);
          y0[it] = load_in<R>(p + S - k0 - k);
          y1[it] = two ? load_in<R>(p + S - k0 - k - 1) : R(0);
        }
      }
    };
    // slabs j of unit u0 + du; one turn more for the epilogue of the last unit
    for (int du = 0, j = 0; ok; ++item) {
      if (item < total) {
        const int op = un.field & t.op_mask;
        const int k0 = t.k0[op], S = t.S[op];
        const R* src = in + ((size_t)un.field * P + (size_t)un.tile * kRowsT) * n;
        const int rows = min(kRowsT, P - un.tile * kRowsT);
        if (item == 0) {
#pragma unroll
          for (int it = 0; it < ITS; ++it) load_row(it, src, rows, kl, k0, S);
        }
        // what these inputs' exponents are lowered by
        struct {
          int x0 = 0, x1 = 0, y0 = 0, y1 = 0;
        } c;
        if constexpr (F64) {
          const unsigned char* e = in_exp[op] + (BWD ? 0 : k0) + min(j * 32 + kl, h);  // (beyond h the inputs are zero)
          c.x0 = e[0], c.x1 = e[1], c.y0 = e[BWD ? h : 0], c.y1 = e[BWD ? h + 1 : 1];
        }
        if (j == 0 && (du == 0 || un.group == 0)) ++tc;
        if (j == 0 && (du == 0 || un.group == 0) && t.nslab == 1) {  // the rows are in the registers
#pragma unroll
          for (int it = 0; it < ITS; ++it) {
            unsigned m = max(max(lowered(magnitude_bits(x0[it]), c.x0), lowered(magnitude_bits(x1[it]), c.x1)),
                             max(lowered(magnitude_bits(y0[it]), c.y0), lowered(magnitude_bits(y1[it]), c.y1)));
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            if ((lane & 15) == 0) row_exp[tc & 3][2 * (kDgWarps * it + cw) + rh] = max((int)(m >> kExpShift), kExpMin);
          }
          __syncwarp();
        } else if (j == 0 && (du == 0 || un.group == 0)) {
          // largest magnitude of each of the warp's rows (FP64: by the high words), 32 loads in flight; a face
          // axis' wall slot holds no input
          constexpr int kRows = 2 * ITS, kStep = sizeof(R) / 4;
          int m[kRows];
#pragma unroll
          for (int r = 0; r < kRows; ++r) m[r] = 0;
          unsigned raw = 0;  // of all rows, not lowered
          const unsigned* w0 = reinterpret_cast<const unsigned*>(src) + (kStep - 1);
#pragma unroll 1
          for (int k = (BWD ? 0 : k0) + lane; k - lane < n; k += 128) {
            unsigned v[4][kRows];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
              for (int r = 0; r < kRows; ++r) {
                const int row = min(2 * (kDgWarps * (r >> 1) + cw) + (r & 1), rows - 1);
                v[q][r] = load_in<R>(w0 + ((size_t)row * n + min(k + 32 * q, n - 1)) * kStep);
              }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int c20 = F64 ? in_exp[op][min(k + 32 * q, n - 1)] << 20 : 0;
#pragma unroll
              for (int r = 0; r < kRows; ++r) {
                const unsigned high = v[q][r] & 0x7fffffffu;
                m[r] = max(m[r], (int)high - c20);
                if (F64) raw = max(raw, high);
              }
            }
          }
          if (F64 && __any_sync(0xffffffffu, raw >= 0x7ff00000u)) {  // an Inf or NaN keeps its exponent: which rows?
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
              const int row = min(2 * (kDgWarps * (r >> 1) + cw) + (r & 1), rows - 1);
              unsigned top = 0;
              for (int k = (BWD ? 0 : k0) + lane; k < n; k += 32)
                top = max(top, load_in<R>(w0 + ((size_t)row * n + k) * kStep) & 0x7fffffffu);
              if (top >= 0x7ff00000u) m[r] = (int)top;
            }
          }
#pragma unroll
          for (int r = 0; r < kRows; ++r) {
            const unsigned top = __reduce_max_sync(0xffffffffu, (unsigned)m[r]);
            if (lane == 0)
              row_exp[tc & 3][2 * (kDgWarps * (r >> 1) + cw) + (r & 1)] = max((int)(top >> kExpShift), kExpMin);
          }
          __syncwarp();
        }
        const int* re = row_exp[tc & 3];
        const int gi = 2 * item, s0 = gi % kSlots, s1 = (gi + 1) % kSlots;
        // the next item: this unit's next slab, or the first of the next unit
        if (j + 1 == t.nslab) nx.step(t);
        const R* nsrc = in + ((size_t)nx.field * P + (size_t)nx.tile * kRowsT) * n;
        const int nrows = item + 1 < total ? min(kRowsT, P - nx.tile * kRowsT) : 0;
        const int nk = (j + 1 == t.nslab ? 0 : (j + 1) * 32) + kl;
        const int nk0 = t.k0[nx.field & t.op_mask], nS = t.S[nx.field & t.op_mask];
        using Val = typename Dg<R>::Val;
        Val i0[ITS], i1[ITS], j0[ITS], j1[ITS];
#pragma unroll
        for (int it = 0; it < ITS; ++it) {
          const int E = re[2 * (kDgWarps * it + cw) + rh];
          i0[it] = scaled(x0[it], E + c.x0);
          i1[it] = scaled(x1[it], E + c.x1);
          j0[it] = scaled(y0[it], E + c.y0);
          j1[it] = scaled(y1[it], E + c.y1);
          load_row(it, nsrc, nrows, nk, nk0, nS);
        }
        // each slot is filled as soon as it is free: with three slots, the MMAs of the slab before run meanwhile
        constexpr int kRow = 2 * kDgWarps * 64;
        const int off = (2 * cw + rh) * 64 + (((kl >> 3) ^ (cw & 3)) << 4) + (kl & 7) * 2;  // row >> 1 = cw mod 4
        // (the warp gives up as one: the shuffles and votes further on take every lane)
        if (gi >= kSlots &&
            !__all_sync(0xffffffffu,
                        mbar_wait(smem_u32(&bar_empty[s0]), ((gi / kSlots) - 1) & 1, t.err, 37, t.spins))) {
          ok = false;
          break;
        }
        unsigned char* dst = smem + s0 * kSlotBytes + off;
#pragma unroll
        for (int it = 0; it < ITS; ++it)
          put_digits(dst + it * kRow, BWD ? i0[it] : i0[it] + j0[it], BWD ? i1[it] : i1[it] + j1[it]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(smem_u32(&bar_conv[s0]));
        if (gi + 1 >= kSlots &&
            !__all_sync(0xffffffffu,
                        mbar_wait(smem_u32(&bar_empty[s1]), (((gi + 1) / kSlots) - 1) & 1, t.err, 38, t.spins))) {
          ok = false;
          break;
        }
        dst = smem + s1 * kSlotBytes + off;
#pragma unroll
        for (int it = 0; it < ITS; ++it)
          put_digits(dst + it * kRow, BWD ? j0[it] : i0[it] - j0[it], BWD ? j1[it] : i1[it] - j1[it]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(smem_u32(&bar_conv[s1]));
      }
      if (j == 0 && du > 0) {  // epilogue of the previous unit
        const int group = pv.group, op = pv.field & t.op_mask, p = pv.tile * kRowsT + erow;
        const bool newer = item < total && un.group == 0;  // tile tc is already the next one
        const bool live = erow < kRowsT && p < P;
        const int k0 = t.k0[op], S = t.S[op];
        R* __restrict__ o = out + (size_t)pv.field * P * n + p;
        R l01 = R(0);
        if (!BWD && t.scale && live) {
          const int a = p / t.nb, b = p - a * t.nb;
          l01 = t.lam[1][op][a] + t.lam[0][op][b] - t.shift[op];
        }
        ok = mbar_wait(smem_u32(&bar_accf), (du - 1) & 1, t.err, 39, t.spins);
        if (!__all_sync(0xffffffffu, ok)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int E = row_exp[(newer ? tc - 1 : tc) & 3][erow];
        const bool bad = E == kExpMax;  // an Inf or NaN among the row's inputs
        // FP32: 2^(E - 140), E in 32 .. 254
        const float row_scale = __uint_as_float((unsigned)(min(E, 254) - 13) << 23);
        const int c1 = __any_sync(0xffffffffu, live) ? min(NC, h - group * NC) : 0;
#pragma unroll 1
        for (int c0 = (cw >> 2) * E_; c0 < c1; c0 += (kDgWarps / 4) * E_) {
          typename Dg<R>::Val vs[E_], va[E_];
          uint32_t rs[ACC][E_], ra[ACC][E_];
#pragma unroll
          for (int d = 0; d < ACC; ++d) tmem_ld(lane_base + d * NC + c0, rs[d]);
#pragma unroll
          for (int d = 0; d < ACC; ++d) tmem_ld(lane_base + 256 + d * NC + c0, ra[d]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int q = 0; q < E_; ++q) vs[q] = join_orders(rs, q), va[q] = join_orders(ra, q);
          if (live) {
            const int j0 = group * NC + c0;
            // rows of the output: modes j and h + j, or cells k0 + j and S - k0 - j
            R* __restrict__ o1 = o + (size_t)(BWD ? k0 + j0 : j0) * P;
            R* __restrict__ o2 = o + (size_t)(BWD ? S - k0 - j0 : h + j0) * P;
#pragma unroll
            for (int q = 0; q < E_; ++q) {
              const int jj = j0 + q;
              if (jj >= h) break;
              R s, a;
              if constexpr (F64) {
                const int e = E + out_exp[op][jj] - 1020;
                const bool fast = e > -1000 && e < 900;
                s = from_fixed(BWD ? vs[q] + va[q] : vs[q], e, fast);
                a = from_fixed(BWD ? vs[q] - va[q] : va[q], e, fast);
              } else {  // both factors are powers of two
                const float col = __int_as_float(out_exp[op][jj]);
                s = (BWD ? vs[q] + va[q] : vs[q]) * col * row_scale;
                a = (BWD ? vs[q] - va[q] : va[q]) * col * row_scale;
              }
              if (bad) s = a = quiet_nan<R>();
              if (BWD) {
                if (k0 + jj <= S - k0 - jj) {  // (an odd face axis has one pair less than h)
                  *o1 = s;
                  *o2 = a;
                }
                if (k0 == 1 && jj == 0) o[0] = R(0);  // the wall slot
                o2 -= P;
              } else {
                if (t.scale) {
                  const R* lz = t.lam[2][op];
                  s = (t.zero_mode && p == 0 && jj == 0) ? R(0) : t.fac[op] * s / (lz[jj] + l01);
                  if (jj < ha) a = t.fac[op] * a / (lz[h + jj] + l01);
                }
                *o1 = s;
                if (jj < ha) *o2 = a;
                o2 += P;
              }
              o1 += P;
            }
          }
        }
        // the accumulators' values are in registers (tcgen05.wait::ld): the MMAs may reuse them
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_acce));
      }
      if (item == total) break;
      if (++j == t.nslab) {
        j = 0;
        ++du;
        pv = un;
        un.step(t);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

template <typename R>
constexpr size_t digit_smem() {
  return (size_t)Dg<R>::kSlots * (Dg<R>::D * kDgDigitBytes + Dg<R>::D * Dg<R>::NC * 64) + 1024;
}

template <typename R>
const HalfDev<R> (&half_of(const fv_grid_s* g))[3][3];
template <>
const HalfDev<double> (&half_of<double>(const fv_grid_s* g))[3][3] { return g->half64; }
template <>
const HalfDev<float> (&half_of<float>(const fv_grid_s* g))[3][3] { return g->half32; }

}  // namespace

template <typename R, int ITS>
static int digit_setup_its() {
  for (auto k : {k_digit_pass<R, false, ITS>, k_digit_pass<R, true, ITS>})
    FV_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)digit_smem<R>()));
  return FV_OK;
}

int digit_setup() {
  static_assert(digit_smem<double>() <= 227 * 1024 && digit_smem<float>() <= 227 * 1024, "ring fits shared memory");
  FV_TRY((digit_setup_its<double, 1>()));
  FV_TRY((digit_setup_its<double, 3>()));
  FV_TRY((digit_setup_its<double, 4>()));
  FV_TRY((digit_setup_its<float, 1>()));
  FV_TRY((digit_setup_its<float, 3>()));
  return digit_setup_its<float, 4>();
}

template <typename R>
int digit_pass(const fv_grid_s* g, int axis, bool bwd, int na, int nb, const int (*kinds)[3], bool per_field,
               const double* sfac, const double* shift, const R* in, R* out, bool scale, bool zero_mode, int nf) {
  const auto& H = half_of<R>(g);
  DgArgs<R> t{};
  t.n = axis == 0 ? g->nx : axis == 1 ? g->ny : g->nz;
  t.P = na * nb;
  t.nb = nb;
  t.op_mask = per_field ? 3 : 0;
  t.scale = scale ? 1 : 0;
  t.zero_mode = zero_mode ? 1 : 0;
  const int h = (t.n + 1) / 2;
  bool cells = true;
  for (int op = 0; op < (per_field ? 4 : 1); ++op) {
    const HalfDev<R>& d = H[axis][kinds[op][axis]];
    t.B[op] = d.dig[bwd ? 1 : 0];
    t.eM[op] = d.dexp[bwd ? 1 : 0];
    t.cM[op] = d.cexp[bwd ? 1 : 0];
    for (int x = 0; x < 3; ++x) t.lam[x][op] = H[x][kinds[op][x]].lam;
    t.fac[op] = (R)sfac[op];
    t.shift[op] = (R)shift[op];
    t.k0[op] = d.k0;
    t.S[op] = d.S;
    cells = cells && d.k0 == 0;
  }
  // pairs of neighbours by one load: rows of an even length from an aligned base, pairs at even offsets
  t.vec = t.n % 2 == 0 && (bwd ? h % 2 == 0 : cells) && (uintptr_t)in % (2 * sizeof(R)) == 0;
  t.groups = (h + Dg<R>::NC - 1) / Dg<R>::NC;
  t.nslab = (h + 31) / 32;
  // Height of the tiles by the workers' time of the busiest SM's units: the conversions of their slabs (which go by the
  // rows) and an epilogue worth about four slabs of 32 rows (which does not).  Fewer rows where a launch has few units.
  int its = 4;
  long long best = -1;
  for (int i : {4, 3, 1}) {
    const int rows = i * 2 * kDgWarps;
    const long long units = (long long)((t.P + rows - 1) / rows) * t.groups * nf;
    const long long cost = (units + g->sms - 1) / g->sms * (i * t.nslab + 4);
    if (best < 0 || cost < best) best = cost, its = i;
  }
  const int rows = its * 2 * kDgWarps;
  t.tiles = (t.P + rows - 1) / rows;
  const long long units = (long long)t.tiles * t.groups * nf;
  if (units > (1LL << 30)) {
    set_error("digit_pass: too many fields in one block");
    return FV_EINVAL;
  }
  t.units = (int)units;
  t.err = g->ws.err;
  t.spins = wait_spins(g);
  const unsigned grid = (unsigned)std::min<long long>(units, g->sms);
  ProfScope ps(g, PROF_TRANSFORM_TC);
  auto go = [&](auto i) {
    constexpr int ITS = decltype(i)::value;
    launch(bwd ? k_digit_pass<R, true, ITS> : k_digit_pass<R, false, ITS>, grid, kDgThreads, digit_smem<R>(), g->stream, t,
           in, out);
  };
  if (its == 4)
    go(std::integral_constant<int, 4>());
  else if (its == 3)
    go(std::integral_constant<int, 3>());
  else
    go(std::integral_constant<int, 1>());
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

template int digit_pass<double>(const fv_grid_s*, int, bool, int, int, const int (*)[3], bool, const double*,
                                const double*, const double*, double*, bool, bool, int);
template int digit_pass<float>(const fv_grid_s*, int, bool, int, int, const int (*)[3], bool, const double*,
                               const double*, const float*, float*, bool, bool, int);

}  // namespace fv
