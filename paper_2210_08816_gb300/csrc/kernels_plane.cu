// Two consecutive half-size passes of a fast-diagonalisation solve (kernels_fdm.cu) in one launch, FP64, small grids.
//
// At these sizes a pass is 1-2 us of FP64 work (two operations per clock and SM) in 4-6 us of launch, first loads and
// drain.  A solve's six passes, forward x, y, z, backward x, y, z, are three pairs of neighbouring axes: (x, y) on
// planes z, (z, x) on planes of a y-mode, (y, z) on planes x.  A cluster of C thread blocks owns a plane of one field:
// block r transforms the rows b of its share of the second axis along the first, writes every result into the shared
// memory of the block that owns its index of the first axis, and, after the cluster's barrier, transforms those rows
// along the second axis and stores them where the plane was (elements keep their place, so that a pair works in place
// and needs no second buffer).  C is what gives every SM a block, at most 4.  The matrices of both axes are loaded before
// the wait for the predecessor.  Every number is formed by the same operations in the same order as by k_half: the
// results agree bit for bit.  Measured: see plane_wins (32^3 J.v + projection 60.2 -> 46.9 us).
#include <cooperative_groups.h>

#include <algorithm>

#include "fv_internal.h"
#include "launch.cuh"

namespace fv {
namespace {

namespace cg = cooperative_groups;
constexpr int kPlThreads = 256;

struct PlaneArgs {
  const double *M1[2][4], *M2[2][4];  // symmetric / antisymmetric matrix per operator, first and second axis
  const double* lam[3][4];            // scaled pair: eigenvalues of the three axes per operator
  double fac[4], shift[4];
  int k1[4], S1[4], k2[4], S2[4];  // first cell and mirror sum of either axis
  int n1, n2, s1, s2, sp, N;       // lengths and strides of the axes, stride of the planes, elements of a field
  int op_mask, scale, zero_mode;
};

struct PlaneShape {
  int h1, h2, rb, rm, la, ly, l2;  // half lengths, rows of a block in either pass, padded leading dimensions
  size_t doubles;
  __host__ __device__ PlaneShape(int n1, int n2, int C) {
    h1 = (n1 + 1) / 2;
    h2 = (n2 + 1) / 2;
    rb = (n2 + C - 1) / C;
    rm = (n1 + C - 1) / C;
    la = rb | 1;
    ly = n2 | 1;
    l2 = rm | 1;
    doubles = 2 * (size_t)h1 * (h1 + 1) + 2 * (size_t)h2 * (h2 + 1) + 2 * (size_t)h1 * la + (size_t)rm * ly +
              2 * (size_t)h2 * l2;
  }
};

// sums over the pairs of one row (column `row` of the k-major A) with row j of the matrices
__device__ __forceinline__ void row_sums(const double* A, int ld, const double* M, int h, int row, int j, double& s,
                                         double& a) {
  const double* a0 = A + row;
  const double* a1 = a0 + h * ld;
  const double* m0 = M + j * (h + 1);
  const double* m1 = m0 + h * (h + 1);
  s = a = 0.0;
#pragma unroll 4
  for (int k = 0; k < h; ++k) {
    s = fma(a0[k * ld], m0[k], s);
    a = fma(a1[k * ld], m1[k], a);
  }
}

template <bool B1, bool B2>
__global__ void __launch_bounds__(kPlThreads) k_plane(const __grid_constant__ PlaneArgs t, const double* in, double* out) {
  extern __shared__ __align__(16) double sm[];
  pdl_begin();
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int plane = blockIdx.x / C, op = (int)blockIdx.y & t.op_mask, tid = threadIdx.x;
  const PlaneShape q(t.n1, t.n2, C);
  const int h1 = q.h1, h2 = q.h2, ha1 = t.n1 / 2, ha2 = t.n2 / 2;
  double* M1 = sm;
  double* M2 = M1 + 2 * h1 * (h1 + 1);
  double* A1 = M2 + 2 * h2 * (h2 + 1);
  double* Y = A1 + 2 * h1 * q.la;
  double* A2 = Y + q.rm * q.ly;
  for (int part = 0; part < 2; ++part) {
    for (int i = tid; i < h1 * h1; i += kPlThreads) {
      const int j = i / h1;
      M1[part * h1 * (h1 + 1) + i + j] = __ldg(t.M1[part][op] + i);
    }
    for (int i = tid; i < h2 * h2; i += kPlThreads) {
      const int j = i / h2;
      M2[part * h2 * (h2 + 1) + i + j] = __ldg(t.M2[part][op] + i);
    }
  }
  cl.sync();  // every block of the cluster is there before any writes into it
  const unsigned ready0 = pdl_wait();
  const size_t at = (size_t)blockIdx.y * t.N + (size_t)plane * t.sp;
  in += ready0 + at;
  out += ready0 + at;

  // first axis
  const int b0 = rank * q.rb, nb = max(min(q.rb, t.n2 - b0), 0);
  const int k1 = t.k1[op], S1 = t.S1[op];
  for (int i = tid; i < nb * h1; i += kPlThreads) {
    int row, k;  // neighbouring threads along the shorter stride
    if (t.s1 < t.s2)
      row = i / h1, k = i - row * h1;
    else
      k = i / nb, row = i - k * nb;
    const double* src = in + (size_t)(b0 + row) * t.s2;
    double s, a;
    if (B1) {
      s = src[(size_t)k * t.s1];
      a = k < ha1 ? src[(size_t)(h1 + k) * t.s1] : 0.0;
    } else {
      const double x = src[(size_t)(k1 + k) * t.s1], y = src[(size_t)(S1 - k1 - k) * t.s1];
      s = x + y;
      a = x - y;
    }
    A1[k * q.la + row] = s;
    A1[(h1 + k) * q.la + row] = a;
  }
  __syncthreads();
  auto put = [&](int i, int b, double v) {  // index i of the first axis, b of the second
    const int owner = i / q.rm;
    cl.map_shared_rank(Y, owner)[(i - owner * q.rm) * q.ly + b] = v;
  };
  for (int i = tid; i < nb * h1; i += kPlThreads) {
    const int j = i / nb, row = i - j * nb, b = b0 + row;
    double s, a;
    row_sums(A1, q.la, M1, h1, row, j, s, a);
    if (B1) {
      const int i1 = k1 + j, i2 = S1 - i1;
      if (i1 <= i2) {  // (an odd face axis has one pair less than h)
        put(i1, b, s + a);
        put(i2, b, s - a);
      }
      if (k1 == 1 && j == 0) put(0, b, 0.0);  // the wall slot
    } else {
      if (t.scale) {  // first axis z, planes of y-modes, rows of x-modes
        const double* lz = t.lam[2][op];
        const double l01 = t.lam[1][op][plane] + t.lam[0][op][b] - t.shift[op];
        s = (t.zero_mode && plane == 0 && b == 0 && j == 0) ? 0.0 : t.fac[op] * s / (lz[j] + l01);
        if (j < ha1) a = t.fac[op] * a / (lz[h1 + j] + l01);
      }
      put(j, b, s);
      if (j < ha1) put(h1 + j, b, a);
    }
  }
  cl.sync();

  // second axis
  const int r0 = rank * q.rm, nm = max(min(q.rm, t.n1 - r0), 0);
  const int k2 = t.k2[op], S2 = t.S2[op];
  for (int i = tid; i < nm * h2; i += kPlThreads) {
    const int row = i / h2, k = i - row * h2;
    const double* src = Y + row * q.ly;
    double s, a;
    if (B2) {
      s = src[k];
      a = k < ha2 ? src[h2 + k] : 0.0;
    } else {
      const double x = src[k2 + k], y = src[S2 - k2 - k];
      s = x + y;
      a = x - y;
    }
    A2[k * q.l2 + row] = s;
    A2[(h2 + k) * q.l2 + row] = a;
  }
  __syncthreads();
  for (int i = tid; i < nm * h2; i += kPlThreads) {
    int row, j;
    if (t.s2 < t.s1)
      row = i / h2, j = i - row * h2;
    else
      j = i / nm, row = i - j * nm;
    double s, a;
    row_sums(A2, q.l2, M2, h2, row, j, s, a);
    double* dst = out + (size_t)(r0 + row) * t.s1;
    if (B2) {
      const int i1 = k2 + j, i2 = S2 - i1;
      if (i1 <= i2) {
        dst[(size_t)i1 * t.s2] = s + a;
        dst[(size_t)i2 * t.s2] = s - a;
      }
      if (k2 == 1 && j == 0) dst[0] = 0.0;
    } else {
      dst[(size_t)j * t.s2] = s;
      if (j < ha2) dst[(size_t)(h2 + j) * t.s2] = a;
    }
  }
}

}  // namespace

// By the multiplications of a half-size pass along the longest axis: three launches win while launches and latencies
// count, and for longer while there are planes enough for the SMs without clusters (the FP64 pipe is as busy then as in
// k_half, whose blocks spread evenly).  Measured (us, six launches of k_half / here): projection of 8^3 29.0 / 17.4,
// 16^3 34.0 / 19.9, 24^3 39.8 / 23.3, 32^3 42.3 / 28.7, 36^3 50.1 / 35.9, 40^3 (1.3e6) 51.8 / 54.2, 48^3 67 / 83 - 105;
// the diffusion solve's four fields 16^3 30.8 / 16.7, 24^3 35.4 / 33.1, 32^3 53.8 / 45.4, 36^3 (3.4e6) 120 / 63,
// 40^3 87 (digits) / 247.  Axes up to 64 cells: both matrices fit beside the rows.
bool plane_wins(const fv_grid_s* g, int nf) {
  const int most = std::max({g->nx, g->ny, g->nz}), least = std::min({g->nx, g->ny, g->nz});
  const bool enough = 2LL * least * nf > g->sms;
  return most <= 64 && (double)g->N * ((most + 1) / 2) * nf <= (enough ? 3.4e6 : 1.2e6);
}

int plane_setup() {
  for (auto k : {k_plane<false, false>, k_plane<false, true>, k_plane<true, true>})
    FV_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  return FV_OK;
}

int plane_solve(const fv_grid_s* g, const int (*kinds)[3], bool per_field, const double* sfac, const double* shift,
                bool zero_mode, const double* in, double* out, int nf) {
  const int len[3] = {g->nx, g->ny, g->nz}, stride[3] = {1, g->nx, g->nx * g->ny};
  for (int pair = 0; pair < 3; ++pair) {
    const int ax1 = pair == 0 ? 0 : pair == 1 ? 2 : 1, ax2 = (ax1 + 1) % 3, axp = (ax1 + 2) % 3;
    const bool b1 = pair == 2, b2 = pair > 0;
    PlaneArgs t{};
    for (int op = 0; op < (per_field ? 4 : 1); ++op) {
      const HalfDev<double>&d1 = g->half64[ax1][kinds[op][ax1]], &d2 = g->half64[ax2][kinds[op][ax2]];
      for (int part = 0; part < 2; ++part) {
        t.M1[part][op] = b1 ? d1.E[part] : d1.F[part];
        t.M2[part][op] = b2 ? d2.E[part] : d2.F[part];
      }
      for (int x = 0; x < 3; ++x) t.lam[x][op] = g->half64[x][kinds[op][x]].lam;
      t.fac[op] = sfac[op];
      t.shift[op] = shift[op];
      t.k1[op] = d1.k0;
      t.S1[op] = d1.S;
      t.k2[op] = d2.k0;
      t.S2[op] = d2.S;
    }
    t.n1 = len[ax1];
    t.n2 = len[ax2];
    t.s1 = stride[ax1];
    t.s2 = stride[ax2];
    t.sp = stride[axp];
    t.N = (int)g->N;
    t.op_mask = per_field ? 3 : 0;
    t.scale = pair == 1 ? 1 : 0;
    t.zero_mode = zero_mode ? 1 : 0;
    const long long planes = (long long)len[axp] * nf;
    // blocks of 128 sums in the first pass at least; clusters of more than four found no room beside the predecessor's
    // blocks (24^3 projection by clusters of 3, 4, 6: 23.4, 24.8, 39.4 us)
    const long long need = ((long long)t.n2 * ((t.n1 + 1) / 2) + 127) / 128;
    const int C = (int)std::max<long long>(std::min<long long>({need, g->sms / planes, 4}), 1);
    // at most one block per SM while there are no more blocks than SMs: an early start beside the predecessor's last
    // blocks must not pile them up (see launch.cuh)
    size_t smem = PlaneShape(t.n1, t.n2, C).doubles * sizeof(double);
    if (planes * C <= g->sms) smem = std::max<size_t>(smem, 120 * 1024);
    void (*k)(PlaneArgs, const double*, double*) =
        pair == 0 ? k_plane<false, false> : pair == 1 ? k_plane<false, true> : k_plane<true, true>;
    ProfScope ps(g, PROF_TRANSFORM);
    launch_cluster(C, k, dim3((unsigned)(len[axp] * C), nf), kPlThreads, smem, g->stream, t, pair == 0 ? in : out, out);
    FV_CUDA(cudaGetLastError());
  }
  return FV_OK;
}

}  // namespace fv
