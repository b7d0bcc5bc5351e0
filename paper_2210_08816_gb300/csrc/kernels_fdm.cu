// Pressure-correction Poisson solve DG phi = rhs by fast diagonalisation (Lynch, Rice & Thomas 1964).
//
// DG is the Kronecker sum A_x (+) A_y (+) A_z of 1D Neumann operators A = W^-1 S (W = diag(widths),
// S symmetric tridiagonal).  With the generalised eigenvectors E (E^T W E = I) and eigenvalues lam,
//     phi = (E_z x E_y x E_x) diag(1 / (lam_x + lam_y + lam_z)) (E_z x E_y x E_x)^-1 rhs,
// the constant mode (all three lam = 0) set to zero.  Each factor is a dense n x n matrix applied along
// one axis: a batched GEMM with K = n.
//
// Rotating passes.  Every pass contracts the CONTIGUOUS axis of its input and writes the mode index as
// the new slowest axis:  in[a][b][k] (k contiguous)  ->  out[m][a][b] = sum_k M[m][k] in[a][b][k].
// Three passes turn (z, y, x) into (x, z, y), (y, x, z) and back to (z, y, x); the forward three map
// cells to modes (the third one divides by Lambda in its epilogue), the backward three map back.  So
// all six are one GEMM shape, C[p][m] = sum_k A[p][k] B[m][k] with both operands k-contiguous, stored
// transposed (out[m][p]).  Tiles BM (p) x BN (m), slabs of BK; thread (tx, ty) owns p = tx + 16 i and
// m = ty + 16 j, so each store instruction writes 16 consecutive p.
#include <type_traits>

#include "fv_internal.h"
#include "launch.cuh"

namespace fv {
namespace {

template <typename R>
struct TileCfg;
template <>
struct TileCfg<float> {
  static constexpr int BM = 128, BN = 128, BK = 32, TM = 8, TN = 8;
};
template <>
struct TileCfg<double> {
  static constexpr int BM = 64, BN = 64, BK = 16, TM = 4, TN = 4;
};

struct PassArgs {
  int P, nm, K;          // rows (a*b), modes, contraction length
  int scale;             // third forward pass: multiply by sfac / (lam_z[m] + lam_y[p / nb] + lam_x[p % nb])
  int nb;
  int zero_mode;         // the (0,0,0) mode is the null space (Neumann): set it to zero
  double sfac;
  double shift;          // scaled pass: sfac / (lam_z + lam_y + lam_x - shift)
};

// (launched without the overlap, so that its input is complete before it starts: the read-only path is open to it)
template <typename R>
__global__ void __launch_bounds__(256) k_transform(PassArgs t, const R* __restrict__ in, const R* __restrict__ M,
                                                    R* __restrict__ out, const R* __restrict__ lx,
                                                    const R* __restrict__ ly, const R* __restrict__ lz) {
  using T = TileCfg<R>;
  pdl_begin();
  const unsigned ready0 = pdl_wait();
  in += ready0;
  out += ready0;
  constexpr int BM = T::BM, BN = T::BN, BK = T::BK, TM = T::TM, TN = T::TN;
  __shared__ R As[BK][BM + 1];
  __shared__ R Bs[BK][BN + 1];
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  const int p0 = blockIdx.x * BM, m0 = blockIdx.y * BN;
  // blockIdx.z: field of a block of fields stored one after another (P x K in, nm x P out)
  in += (size_t)blockIdx.z * t.P * t.K;
  out += (size_t)blockIdx.z * t.nm * t.P;
  R acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = R(0);

  for (int k0 = 0; k0 < t.K; k0 += BK) {
#pragma unroll
    for (int e = tid; e < BM * BK; e += 256) {
      const int kk = e % BK, rr = e / BK;
      const int p = p0 + rr, k = k0 + kk;
      As[kk][rr] = (p < t.P && k < t.K) ? in[(long long)p * t.K + k] : R(0);
    }
#pragma unroll
    for (int e = tid; e < BN * BK; e += 256) {
      const int kk = e % BK, cc = e / BK;
      const int m = m0 + cc, k = k0 + kk;
      Bs[kk][cc] = (m < t.nm && k < t.K) ? M[(long long)m * t.K + k] : R(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      R a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][tx + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][ty + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int m = m0 + ty + 16 * j;
    if (m >= t.nm) continue;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int p = p0 + tx + 16 * i;
      if (p >= t.P) continue;
      R val = acc[i][j];
      if (t.scale) {
        const int a = p / t.nb, b = p - a * t.nb;
        val = (t.zero_mode && m == 0 && a == 0 && b == 0) ? R(0) : R(t.sfac) * val / (lz[m] + ly[a] + lx[b] - R(t.shift));
      }
      out[(long long)m * t.P + p] = val;
    }
  }
}

// The passes of a mirror-symmetric grid on the CUDA cores: every 1D operator splits into a symmetric and an
// antisymmetric half (see HalfOpHost), so that a pass contracts the sums and differences of mirrored inputs
// with two h x h matrices, half the multiplications of the dense form.
//
// A CTA owns 32 rows p (one per lane: the rotated store writes 32 consecutive p) and 4 U mode or cell pairs;
// warp w holds the accumulators of pairs U w .. U w + U - 1, symmetric and antisymmetric.  Slabs of 32 inputs
// pairs are staged k-major (padded rows: no bank conflicts), the matrix slabs beside them are read as
// broadcasts.  The FP64 form is bound by the FP64 pipe (two operations per clock and SM: 8 warps cover it), so
// what matters is that the CTAs spread over all SMs: U falls from 4 to 1 until the launch has two CTAs per SM.
// blockIdx.z: field of a block of fields stored one after another; with op_mask 3 field f uses operator f (the
// diffusion solve), with 0 all use operator 0.
constexpr int kHalfK = 32;

template <typename R>
struct HalfArgs {
  const R* M[2][4];    // symmetric / antisymmetric matrix per operator
  const R* lam[3][4];  // scaled pass: eigenvalues of the three axes per operator
  R fac[4], shift[4];  // scaled pass: fac / (lam_z + lam_y + lam_x - shift)
  int k0[4], S[4];
  int P, n, nb, op_mask, scale, zero_mode;
};

template <typename R, bool BWD, int U>
__global__ void __launch_bounds__(128) k_half(const __grid_constant__ HalfArgs<R> t, const R* in,
                                               R* __restrict__ out) {
  pdl_begin();
  const unsigned ready0 = pdl_wait();
  in += ready0;
  out += ready0;
  constexpr int UB = 4 * U, V = 16 / sizeof(R);
  using Vec = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
  __shared__ R As[2][kHalfK][33];
  __shared__ __align__(16) R Bs[2][UB][kHalfK];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = t.n, P = t.P, h = (n + 1) / 2, ha = n / 2;
  const int op = (int)blockIdx.z & t.op_mask;
  const int p0 = blockIdx.x * 32, j0 = blockIdx.y * UB;
  const int k0 = t.k0[op], S = t.S[op];
  const R* Ms = t.M[0][op];
  const R* Ma = t.M[1][op];
  in += (size_t)blockIdx.z * P * n;
  out += (size_t)blockIdx.z * P * n;
  R acc[2][U];
#pragma unroll
  for (int u = 0; u < U; ++u) acc[0][u] = acc[1][u] = R(0);
  for (int kc = 0; kc < h; kc += kHalfK) {
    const int k = kc + lane;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int row = warp + 4 * r, p = p0 + row;
      R s = R(0), a = R(0);
      if (p < P && k < h) {
        const R* src = in + (size_t)p * n;
        if (BWD) {
          s = src[k];
          a = k < ha ? src[h + k] : R(0);
        } else {
          const R x = src[k0 + k], y = src[S - k0 - k];
          s = x + y;
          a = x - y;
        }
      }
      As[0][lane][row] = s;
      As[1][lane][row] = a;
    }
#pragma unroll
    for (int u = warp; u < UB; u += 4) {
      const bool in_m = j0 + u < h && k < h;
      Bs[0][u][lane] = in_m ? Ms[(size_t)(j0 + u) * h + k] : R(0);
      Bs[1][u][lane] = in_m ? Ma[(size_t)(j0 + u) * h + k] : R(0);
    }
    __syncthreads();
    const int kn = min(kHalfK, (h - kc + V - 1) / V * V);  // the slab is zero-filled beyond h
    for (int kk = 0; kk < kn; kk += V) {
      R a0[V], a1[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        a0[v] = As[0][kk + v][lane];
        a1[v] = As[1][kk + v][lane];
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const Vec b0 = *reinterpret_cast<const Vec*>(&Bs[0][warp * U + u][kk]);
        const Vec b1 = *reinterpret_cast<const Vec*>(&Bs[1][warp * U + u][kk]);
        const R* e0 = reinterpret_cast<const R*>(&b0);
        const R* e1 = reinterpret_cast<const R*>(&b1);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          acc[0][u] = fma(a0[v], e0[v], acc[0][u]);
          acc[1][u] = fma(a1[v], e1[v], acc[1][u]);
        }
      }
    }
    __syncthreads();
  }
  const int p = p0 + lane;
  if (p >= P) return;
  R l01 = R(0);
  bool null_row = false;
  if (!BWD && t.scale) {
    const int a = p / t.nb, b = p - a * t.nb;
    l01 = t.lam[1][op][a] + t.lam[0][op][b] - t.shift[op];
    null_row = t.zero_mode && p == 0;
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int j = j0 + warp * U + u;
    if (j >= h) break;
    R s = acc[0][u], a = acc[1][u];
    if (BWD) {
      const int i1 = k0 + j, i2 = S - i1;
      if (i1 <= i2) {  // (an odd face axis has one pair less than h)
        out[(size_t)i1 * P + p] = s + a;
        out[(size_t)i2 * P + p] = s - a;
      }
      if (k0 == 1 && j == 0) out[p] = R(0);  // the wall slot
    } else {
      if (t.scale) {
        const R* lz = t.lam[2][op];
        s = (null_row && j == 0) ? R(0) : t.fac[op] * s / (lz[j] + l01);
        if (j < ha) a = t.fac[op] * a / (lz[h + j] + l01);
      }
      out[(size_t)j * P + p] = s;
      if (j < ha) out[(size_t)(h + j) * P + p] = a;
    }
  }
}

template <typename R>
const HalfDev<R> (&half_of(const fv_grid_s* g))[3][3];
template <>
const HalfDev<double> (&half_of<double>(const fv_grid_s* g))[3][3] { return g->half64; }
template <>
const HalfDev<float> (&half_of<float>(const fv_grid_s* g))[3][3] { return g->half32; }

// Digit products on the tensor cores (kernels_digit.cu) instead of the CUDA-core form, by the multiplications of a
// half-size pass: a digit pass has a floor of ~6 us (FP64 ~11) before its length shows.  Measured (us a projection, CUDA
// cores / digits): FP64 40^3 (1.4e6) 53 / 69, 44^3 65 / 70, 48^3 (2.8e6) 75 / 72, 52^3 (3.9e6) 104 / 77, 56^3 109 / 79;
// FP32 50^3 29 / 33, 60^3 37.5 / 42, 70^3 (1.2e7) 45 / 51, 80^3 (2.1e7) 55 / 57, 86^3 (2.8e7) 56 / 55.5, 90^3 63 / 57; the
// diffusion solve's four fields in FP32 50^3 (1.3e7) 31.8 / 32.9, 52^3 (1.5e7) 31.6 / 33.1, 56^3 (2.1e7) 34.7 / 33.2, 60^3
// 42 / 36, 80^3 100 / 81.  The number of vectors in a block does not count: a block's results are those of its vectors one
// by one, bit for bit.
template <typename R>
bool digit_wins(int n, long long rows) {
  return (double)rows * n * ((n + 1) / 2) >= (sizeof(R) == 8 ? kDigitWork64 : kDigitWork32);
}

// Unused shared memory that leaves room for `per` blocks on an SM, all of it or (FP32, whose launches are short) no more than
// that takes.
template <typename R>
constexpr int half_pad(int U, int per) {
  return (sizeof(R) == 8 ? 222 * 1024 / per : 228 * 1024 / (per + 1) + 1024) -
         (int)(sizeof(R) * (2 * kHalfK * 33 + 2 * 4 * U * kHalfK)) - (sizeof(R) == 8 ? 1024 : 0);
}

template <typename R, int U>
int half_setup_u() {
  for (auto k : {k_half<R, false, U>, k_half<R, true, U>})
    FV_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, half_pad<R>(U, 1)));
  return FV_OK;
}

// One pass along `axis` over nf fields of a (na x nb) x n block, kinds[op][axis] = the operators (one, or four
// with per_field): in[a][b][k] -> out[m][a][b] with the modes in the half order.
template <typename R>
int half_pass(const fv_grid_s* g, int axis, bool bwd, int na, int nb, const int (*kinds)[3], bool per_field,
              const double* sfac, const double* shift, const R* in, R* out, bool scale, bool zero_mode, int nf) {
  const int len = axis == 0 ? g->nx : axis == 1 ? g->ny : g->nz;
  if (g->digit_ready && digit_wins<R>(len, (long long)na * nb * (per_field ? 4 : 1)))
    return digit_pass<R>(g, axis, bwd, na, nb, kinds, per_field, sfac, shift, in, out, scale, zero_mode, nf);
  const auto& H = half_of<R>(g);
  HalfArgs<R> t{};
  t.n = axis == 0 ? g->nx : axis == 1 ? g->ny : g->nz;
  t.P = na * nb;
  t.nb = nb;
  t.op_mask = per_field ? 3 : 0;
  t.scale = scale ? 1 : 0;
  t.zero_mode = zero_mode ? 1 : 0;
  for (int op = 0; op < (per_field ? 4 : 1); ++op) {
    const HalfDev<R>& d = H[axis][kinds[op][axis]];
    for (int part = 0; part < 2; ++part) t.M[part][op] = bwd ? d.E[part] : d.F[part];
    for (int x = 0; x < 3; ++x) t.lam[x][op] = H[x][kinds[op][x]].lam;
    t.fac[op] = (R)sfac[op];
    t.shift[op] = (R)shift[op];
    t.k0[op] = d.k0;
    t.S[op] = d.S;
  }
  const int h = (t.n + 1) / 2;
  const long long rows = (long long)((t.P + 31) / 32) * nf;
  const int U = rows * ((h + 15) / 16) >= 2 * g->sms ? 4 : rows * ((h + 7) / 8) >= 2 * g->sms ? 2 : 1;
  const dim3 grid((t.P + 31) / 32, (h + 4 * U - 1) / (4 * U), nf);
  ProfScope ps(g, PROF_TRANSFORM);
  void (*k)(HalfArgs<R>, const R*, R*);
  if (bwd)
    k = U == 4 ? k_half<R, true, 4> : U == 2 ? k_half<R, true, 2> : k_half<R, true, 1>;
  else
    k = U == 4 ? k_half<R, false, 4> : U == 2 ? k_half<R, false, 2> : k_half<R, false, 1>;
  // One block per SM, or two, ...: unused shared memory keeps more from being placed there, so that the launch can overlap
  // its predecessor and still spread evenly: 32^3 FP64 J.v + projection 73 us without the overlap, 58.5 so; FP32 projection of
  // 800 x 16 x 16 113 us with the overlap alone, 90 so, 60^3 41.3 and 36.5.  From seven blocks per SM on FP64 passes go
  // without the overlap and FP32 ones, whose blocks leave each other room, without the padding.
  const long long per = ((long long)grid.x * grid.y * grid.z + g->sms - 1) / g->sms;
  if (per <= 6)
    launch(k, grid, 128, half_pad<R>(U, (int)per), g->stream, t, in, out);
  else
    launch(sizeof(R) == 4, k, grid, 128, 0, g->stream, t, in, out);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

// the six passes over nf fields: in -> out, tmp of the same size (out may alias in)
template <typename R>
int half_solve(const fv_grid_s* g, const int (*kinds)[3], bool per_field, const double* sfac, const double* shift,
               bool zero_mode, const R* in, R* out, R* tmp, int nf) {
  const int nx = g->nx, ny = g->ny, nz = g->nz;
  if (nf < 1 || nf > 65535) {
    set_error("half_solve: number of fields out of range");
    return FV_EINVAL;
  }
  if constexpr (sizeof(R) == 8) {
    if (plane_wins(g, nf)) return plane_solve(g, kinds, per_field, sfac, shift, zero_mode, in, out, nf);
  }
  // forward: (z,y,x) -> (mx,z,y) -> (my,mx,z) -> (mz,my,mx) / Lambda; backward the same way round
  FV_TRY(half_pass<R>(g, 0, false, nz, ny, kinds, per_field, sfac, shift, in, tmp, false, zero_mode, nf));
  FV_TRY(half_pass<R>(g, 1, false, nx, nz, kinds, per_field, sfac, shift, tmp, out, false, zero_mode, nf));
  FV_TRY(half_pass<R>(g, 2, false, ny, nx, kinds, per_field, sfac, shift, out, tmp, true, zero_mode, nf));
  FV_TRY(half_pass<R>(g, 0, true, nz, ny, kinds, per_field, sfac, shift, tmp, out, false, zero_mode, nf));
  FV_TRY(half_pass<R>(g, 1, true, nx, nz, kinds, per_field, sfac, shift, out, tmp, false, zero_mode, nf));
  return half_pass<R>(g, 2, true, ny, nx, kinds, per_field, sfac, shift, tmp, out, false, zero_mode, nf);
}

constexpr int kPoissonKinds[1][3] = {{HALF_NEUMANN, HALF_NEUMANN, HALF_NEUMANN}};
// fields u, v, w: face-centred along the own axis, cell-centred Dirichlet across; T: Dirichlet in x only
constexpr int kDiffusionKinds[4][3] = {{HALF_FACE, HALF_CELL, HALF_CELL},
                                       {HALF_CELL, HALF_FACE, HALF_CELL},
                                       {HALF_CELL, HALF_CELL, HALF_FACE},
                                       {HALF_CELL, HALF_NEUMANN, HALF_NEUMANN}};

template <typename R>
const FdmDev<R>& fdm_of(const fv_grid_s* g);
template <>
const FdmDev<double>& fdm_of<double>(const fv_grid_s* g) { return g->fdm64; }
template <>
const FdmDev<float>& fdm_of<float>(const fv_grid_s* g) { return g->fdm32; }

// in[a][b][k] -> out[m][a][b] with M (nm x K); a scaled pass divides by the eigenvalue sums of lam[0..2]
template <typename R>
int pass_ops(const fv_grid_s* g, const R* M, int na, int nb, int K, const R* in, R* out, bool scale,
             const R* const lam[3], bool zero_mode, double sfac, int nvec = 1, double shift = 0.0) {
  using T = TileCfg<R>;
  PassArgs t{};
  t.P = na * nb;
  t.nm = K;
  t.K = K;
  t.scale = scale ? 1 : 0;
  t.nb = nb;
  t.zero_mode = zero_mode ? 1 : 0;
  t.sfac = sfac;
  t.shift = shift;
  dim3 grid((t.P + T::BM - 1) / T::BM, (t.nm + T::BN - 1) / T::BN, nvec);
  ProfScope ps(g, PROF_TRANSFORM);
  launch_spread(k_transform<R>, grid, 256, 0, g->stream, t, in, M, out, lam[0], lam[1], lam[2]);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

template <typename R>
int pass(const fv_grid_s* g, const R* M, int na, int nb, int K, const R* in, R* out, bool scale, int nvec = 1) {
  const FdmDev<R>& f = fdm_of<R>(g);
  return pass_ops<R>(g, M, na, nb, K, in, out, scale, f.lam, true, 1.0, nvec);
}

template <typename R>
const FdmDev<R>& cd_of(const fv_grid_s* g);
template <>
const FdmDev<double>& cd_of<double>(const fv_grid_s* g) { return g->cd64; }
template <>
const FdmDev<float>& cd_of<float>(const fv_grid_s* g) { return g->cd32; }
template <typename R>
const FdmDev<R>& fd_of(const fv_grid_s* g);
template <>
const FdmDev<double>& fd_of<double>(const fv_grid_s* g) { return g->fd64; }
template <>
const FdmDev<float>& fd_of<float>(const fv_grid_s* g) { return g->fd32; }

}  // namespace

int half_setup() {
  FV_TRY((half_setup_u<double, 1>()));
  FV_TRY((half_setup_u<double, 2>()));
  FV_TRY((half_setup_u<double, 4>()));
  FV_TRY((half_setup_u<float, 1>()));
  FV_TRY((half_setup_u<float, 2>()));
  return half_setup_u<float, 4>();
}

template <typename R>
int launch_poisson_block(const fv_grid_s* g, const R* rhs, R* phi, R* tmp, int nvec) {
  const int nx = g->nx, ny = g->ny, nz = g->nz;
  if (nvec < 1 || nvec > 65535) {
    set_error("launch_poisson_block: nvec out of range");
    return FV_EINVAL;
  }
  if constexpr (sizeof(R) == 4) {
    if (g->tc_ready) {  // the tensor-core passes over the stacked fields
      unsigned* slots = fmax_slots(g, nvec);
      FV_TRY(tc_pass(g, 0, nz, ny, rhs, tmp, slots, nvec));
      FV_TRY(tc_pass(g, 1, nx, nz, tmp, phi, slots, nvec));
      FV_TRY(tc_pass(g, 2, ny, nx, phi, tmp, slots, nvec));
      FV_TRY(tc_pass(g, 3, nz, ny, tmp, phi, slots, nvec));
      FV_TRY(tc_pass(g, 4, nx, nz, phi, tmp, slots, nvec));
      return tc_pass(g, 5, ny, nx, tmp, phi, slots, nvec);
    }
  }
  if (g->half_ready) {
    const double one = 1.0, zero = 0.0;
    return half_solve<R>(g, kPoissonKinds, false, &one, &zero, true, rhs, phi, tmp, nvec);
  }
  // dense passes, forward: (z,y,x) -> (mx,z,y) -> (my,mx,z) -> (mz,my,mx) / Lambda
  const FdmDev<R>& f = fdm_of<R>(g);
  FV_TRY(pass<R>(g, f.Einv[0], nz, ny, nx, rhs, tmp, false, nvec));
  FV_TRY(pass<R>(g, f.Einv[1], nx, nz, ny, tmp, phi, false, nvec));
  FV_TRY(pass<R>(g, f.Einv[2], ny, nx, nz, phi, tmp, true, nvec));
  // backward: (mz,my,mx) -> (x,mz,my) -> (y,x,mz) -> (z,y,x)
  FV_TRY(pass<R>(g, f.E[0], nz, ny, nx, tmp, phi, false, nvec));
  FV_TRY(pass<R>(g, f.E[1], nx, nz, ny, phi, tmp, false, nvec));
  FV_TRY(pass<R>(g, f.E[2], ny, nx, nz, tmp, phi, false, nvec));
  return FV_OK;
}

template <typename R>
int launch_poisson(const fv_grid_s* g, const R* rhs, R* phi, R* tmp) {
  return launch_poisson_block<R>(g, rhs, phi, tmp, 1);
}

template int launch_poisson<float>(const fv_grid_s*, const float*, float*, float*);
template int launch_poisson<double>(const fv_grid_s*, const double*, double*, double*);
template int launch_poisson_block<double>(const fv_grid_s*, const double*, double*, double*, int);
template int launch_poisson_block<float>(const fv_grid_s*, const float*, float*, float*, int);

// Diffusion operator of one field, L_f = s_f (L_x (+) L_y (+) L_z), inverted like the pressure operator:
// velocity component c uses the face-centred Dirichlet operator along its own axis and the cell-centred
// Dirichlet operator across (no-slip walls half a cell away); temperature uses cell-centred Dirichlet in
// x (Eq. 4, homogeneous) and the Neumann operator in y and z (Eqs. 5-6), with s_T = 1/Pr.  No zero mode.
// s != 0: (L_f - s I)^-1 instead (the eigenvalues of L_f are (lam_x + lam_y + lam_z) / s_f).
// On mirror-symmetric grids the four fields go through each pass together (6 launches instead of 24).
template <typename R>
int launch_diffusion_solve(const fv_grid_s* g, const R* in, R* out, R* tmp, double s) {
  const int nx = g->nx, ny = g->ny, nz = g->nz;
  if (g->half_ready) {
    const double sfac[4] = {1.0, 1.0, 1.0, g->Pr}, shift[4] = {s, s, s, s * g->Pr};
    return half_solve<R>(g, kDiffusionKinds, true, sfac, shift, false, in, out, tmp, 4);
  }
  for (int f = 0; f < 4; ++f) {
    const FdmDev<R>* op[3];
    for (int d = 0; d < 3; ++d) {
      if (f < 3)
        op[d] = (d == f) ? &fd_of<R>(g) : &cd_of<R>(g);
      else
        op[d] = (d == 0) ? &cd_of<R>(g) : &fdm_of<R>(g);
    }
    const R* lam[3] = {op[0]->lam[0], op[1]->lam[1], op[2]->lam[2]};
    const double sfac = (f == 3) ? g->Pr : 1.0;
    const R* fi = in + (size_t)f * g->N;
    R* fo = out + (size_t)f * g->N;
    FV_TRY(pass_ops<R>(g, op[0]->Einv[0], nz, ny, nx, fi, tmp, false, lam, false, 1.0));
    FV_TRY(pass_ops<R>(g, op[1]->Einv[1], nx, nz, ny, tmp, fo, false, lam, false, 1.0));
    FV_TRY(pass_ops<R>(g, op[2]->Einv[2], ny, nx, nz, fo, tmp, true, lam, false, sfac, 1, s * sfac));
    FV_TRY(pass_ops<R>(g, op[0]->E[0], nz, ny, nx, tmp, fo, false, lam, false, 1.0));
    FV_TRY(pass_ops<R>(g, op[1]->E[1], nx, nz, ny, fo, tmp, false, lam, false, 1.0));
    FV_TRY(pass_ops<R>(g, op[2]->E[2], ny, nx, nz, tmp, fo, false, lam, false, 1.0));
  }
  return FV_OK;
}

template int launch_diffusion_solve<double>(const fv_grid_s*, const double*, double*, double*, double);
template int launch_diffusion_solve<float>(const fv_grid_s*, const float*, float*, float*, double);

}  // namespace fv
