// Host side of the digit passes (kernels_digit.cu): the half-size matrices of an axis operator as balanced base-256
// digits in FP16, in the blocks and the shared-memory layout that the kernel copies.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "fv_internal.h"

namespace fv {

// FP16 bits of an integer of magnitude <= 128 (exact)
static uint16_t half_bits(int v) {
  if (v == 0) return 0;
  const unsigned m = (unsigned)std::abs(v);
  int e = 0;
  while ((m >> e) > 1) ++e;
  return (uint16_t)((v < 0 ? 0x8000u : 0u) | ((unsigned)(e + 15) << 10) | ((m << (10 - e)) & 0x3ffu));
}

void build_digits(const std::vector<double> (&M)[2], int h, int D, int NC, std::vector<unsigned char>& blocks,
                  std::vector<int>& exps) {
  const int groups = (h + NC - 1) / NC, nslab = (h + 31) / 32;
  const size_t block = (size_t)D * NC * 64;
  exps.assign(h, 0);
  for (int j = 0; j < h; ++j) {
    double top = 0.0;
    for (int part = 0; part < 2; ++part)
      for (int k = 0; k < h; ++k) top = std::max(top, std::fabs(M[part][(size_t)j * h + k]));
    int q = 0;
    if (top > 0.0) std::frexp(top, &q);  // top < 2^q
    exps[j] = q - (8 * D - 1);           // integers of magnitude <= 2^(8 D - 1)
  }
  blocks.assign(block * 2 * groups * nslab, 0);
  for (int part = 0; part < 2; ++part)
    for (int j = 0; j < h; ++j)
      for (int k = 0; k < h; ++k) {
        long long J = std::llrint(std::ldexp(M[part][(size_t)j * h + k], -exps[j]));
        unsigned char* b = blocks.data() + ((size_t)(part * groups + j / NC) * nslab + k / 32) * block;
        for (int i = D - 1; i >= 0; --i) {
          const int dgt = i == 0 ? (int)J : (int)(((J + 128) & 255) - 128);
          J = (J - dgt) >> 8;
          // row r of the stacked operand, 64-byte swizzled: 16-byte chunk c at c ^ ((r >> 1) & 3)
          const int r = i * NC + j % NC, kk = k % 32, c = (kk >> 3) ^ ((r >> 1) & 3);
          const uint16_t v = half_bits(dgt);
          std::memcpy(b + (size_t)r * 64 + c * 16 + (kk & 7) * 2, &v, 2);
        }
      }
}

}  // namespace fv
