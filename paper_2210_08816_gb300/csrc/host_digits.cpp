// Host side of the digit passes (kernels_digit.cu): the half-size matrices of an axis operator as balanced base-256
// digits in FP16, in the blocks and the shared-memory layout that the kernel copies.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "fv_internal.h"

namespace fv {

bool tc_sizes(const int n[3]) {
  for (int d = 0; d < 3; ++d)
    if (n[d] < 32 || n[d] > 256 || n[d] % 32 != 0) return false;
  return true;
}

bool digits_reached(const int n[3], int prec) {
  const double work = 4.0 * n[0] * n[1] * n[2] * ((std::max({n[0], n[1], n[2]}) + 1) / 2);
  return prec == 0 ? work >= kDigitWork64 : work >= kDigitWork32 || tc_sizes(n);
}

// FP16 bits of the integers -128 .. 128 (exact)
struct HalfTable {
  uint16_t bits[257];
  HalfTable() {
    for (int v = -128; v <= 128; ++v) {
      const unsigned m = (unsigned)std::abs(v);
      int e = 0;
      while ((m >> e) > 1) ++e;
      bits[v + 128] = m == 0 ? 0
                             : (uint16_t)((v < 0 ? 0x8000u : 0u) | ((unsigned)(e + 15) << 10) | ((m << (10 - e)) & 0x3ffu));
    }
  }
};

// Largest magnitude of row j of both parts as the exponent q with |entries| < 2^q
static int row_exponent(const std::vector<double> (&M)[2], int h, int j) {
  double top = 0.0;
  for (int part = 0; part < 2; ++part)
    for (int k = 0; k < h; ++k) top = std::max(top, std::fabs(M[part][(size_t)j * h + k]));
  int q = 0;
  if (top > 0.0) std::frexp(top, &q);
  return q;
}

// Offset, in halves, of column k of row r of a block: 64-byte rows, 16-byte chunk c at c ^ ((r >> 1) & 3)
static inline size_t swizzled(int r, int kk) { return (size_t)r * 32 + (((kk >> 3) ^ ((r >> 1) & 3)) << 3) + (kk & 7); }

void build_digits(const std::vector<double> (&M)[2], int h, int D, int NC, bool shared, std::vector<unsigned char>& blocks,
                  std::vector<int>& exps, std::vector<unsigned char>& cexps) {
  static const HalfTable table;
  const int groups = (h + NC - 1) / NC, nslab = (h + 31) / 32;
  const size_t block = (size_t)D * NC * 32;  // halves
  blocks.assign(block * 2 * groups * nslab * 2, 0);
  uint16_t* out = reinterpret_cast<uint16_t*>(blocks.data());
  exps.assign(h, 0);
  cexps.assign(2 * (size_t)h, 0);
  std::vector<int> q(2 * (size_t)h, INT_MIN);  // exponent of every column's largest magnitude
  std::vector<double> most(h);
  int top = INT_MIN;
  for (int part = 0; part < 2; ++part) {
    std::fill(most.begin(), most.end(), 0.0);
    for (int j = 0; j < h; ++j)
      for (int k = 0; k < h; ++k) most[k] = std::max(most[k], std::fabs(M[part][(size_t)j * h + k]));
    for (int k = 0; k < h; ++k) {
      if (most[k] > 0.0) std::frexp(most[k], &q[part * h + k]);
      top = std::max(top, q[part * h + k]);
    }
  }
  for (int k = 0; k < h && shared; ++k) q[k] = q[h + k] = std::max(q[k], q[h + k]);
  for (size_t i = 0; i < q.size(); ++i)
    if (q[i] != INT_MIN) cexps[i] = (unsigned char)std::min(top - q[i], kDigitMaxColumn);
  std::vector<double> S[2];  // the columns scaled (powers of two: exact)
  for (int part = 0; part < 2; ++part) {
    std::vector<double> scale(h);
    for (int k = 0; k < h; ++k) scale[k] = std::ldexp(1.0, cexps[part * h + k]);
    S[part].resize((size_t)h * h);
    for (int j = 0; j < h; ++j)
      for (int k = 0; k < h; ++k) S[part][(size_t)j * h + k] = M[part][(size_t)j * h + k] * scale[k];
  }
  for (int j = 0; j < h; ++j) {
    exps[j] = row_exponent(S, h, j) - (8 * D - 1);  // integers of magnitude <= 2^(8 D - 1)
    const double scale = std::ldexp(1.0, -exps[j]);
    for (int part = 0; part < 2; ++part)
      for (int k = 0; k < h; ++k) {
        long long J = std::llrint(S[part][(size_t)j * h + k] * scale);
        uint16_t* b = out + ((size_t)(part * groups + j / NC) * nslab + k / 32) * block;
        for (int i = D - 1; i >= 0; --i) {
          const int dgt = i == 0 ? (int)J : (int)(((J + 128) & 255) - 128);
          J = (J - dgt) >> 8;
          b[swizzled(i * NC + j % NC, k % 32)] = table.bits[dgt + 128];
        }
      }
  }
}

// FP16 rounding of |v| < 65520 (nearest even, subnormals included): the value and its bits
static double round_half(double v, uint16_t& bits) {
  uint64_t u;
  std::memcpy(&u, &v, 8);
  const int e = std::max((int)((u >> 52) & 0x7ff) - 1023, -14);
  uint64_t unit = (uint64_t)(e - 10 + 1023) << 52, inverse = (uint64_t)(10 - e + 1023) << 52;
  double un, in;
  std::memcpy(&un, &unit, 8);
  std::memcpy(&in, &inverse, 8);
  const long long m = std::llrint(std::fabs(v) * in);  // in units of 2^(e - 10)
  // m = 2048 carries into the exponent field, m < 1024 is subnormal
  bits = (uint16_t)((v < 0 ? 0x8000u : 0u) | (m == 0 ? 0u : ((unsigned)(e + 14) << 10) + (unsigned)m));
  const double r = (double)m * un;
  return v < 0 ? -r : r;
}

void build_halves(const std::vector<double> (&M)[2], int h, int NC, std::vector<unsigned char>& blocks,
                  std::vector<int>& exps) {
  const int groups = (h + NC - 1) / NC, nslab = (h + 31) / 32;
  const size_t block = (size_t)2 * NC * 32;  // halves
  exps.assign(h, 0);
  blocks.assign(block * 2 * groups * nslab * 2, 0);
  uint16_t* out = reinterpret_cast<uint16_t*>(blocks.data());
  for (int j = 0; j < h; ++j) {
    exps[j] = row_exponent(M, h, j) - 14;  // scaled below 2^14
    const double scale = std::ldexp(1.0, -exps[j]);
    for (int part = 0; part < 2; ++part)
      for (int k = 0; k < h; ++k) {
        const double x = M[part][(size_t)j * h + k] * scale;
        uint16_t v[2];
        const double hi = round_half(x, v[0]);
        round_half(x - hi, v[1]);
        uint16_t* b = out + ((size_t)(part * groups + j / NC) * nslab + k / 32) * block;
        for (int i = 0; i < 2; ++i) b[swizzled(i * NC + j % NC, k % 32)] = v[i];
      }
  }
}

}  // namespace fv
