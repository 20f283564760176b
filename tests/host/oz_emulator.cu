// Host run of the exact tensor-core block's arithmetic (test only): digits of
// a row and of a matrix, the kept digit products summed by weight as exact
// integers, and the join, against long double.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_2106_13995_gb300/csrc/oz_digits.cuh"
#include "../../paper_2106_13995_gb300/csrc/sv_internal.h"

using namespace sv;

static double half_value(uint16_t h) {
  const int e = (h >> 10) & 31, m = h & 1023;
  const double v = e ? std::ldexp(1024.0 + m, e - 25) : std::ldexp((double)m, -24);
  return (h & 0x8000) ? -v : v;
}

// out = U x (32 complex numbers each, interleaved) through the digits; worst[0]:
// the largest error over the row's norm, worst[1]: the largest sum of weight at
// most 4.  Returns 0, 1 when the matrix does not qualify, or -1.
extern "C" int oz_block(const double *u, const double *x, double *out, double *worst) {
  std::vector<cd> U(32 * 32);
  for (int i = 0; i < 32 * 32; i++) U[i] = cd(u[2 * i], u[2 * i + 1]);
  std::vector<uint16_t> B;
  int eu = 0;
  if (!oz_pack_matrix(U, B, eu)) return 1;
  uint32_t E = 1, hi[64], lo[64];
  for (int k = 0; k < 64; k++) {
    uint64_t b;
    std::memcpy(&b, &x[k], 8);
    hi[k] = (uint32_t)(b >> 32);
    lo[k] = (uint32_t)b;
    E = std::max(E, oz_exponent(hi[k]));
  }
  uint64_t w[64];
  long double norm = 0;
  for (int k = 0; k < 64; k++) {
    w[k] = oz_fields(hi[k], lo[k], E);
    norm += (long double)x[k] * x[k];
    for (int i = 0; i < kOzDigits; i++)
      if (std::abs(oz_digit(w[k], i)) > 256) return -1;
  }
  norm = std::sqrt(norm);
  worst[0] = worst[1] = 0;
  for (int n = 0; n < 64; n++) {
    float l[kOzDigits];
    for (int s = 0; s < kOzDigits; s++) {
      int64_t sum = 0;
      for (int i = 0; i <= s; i++)
        for (int k = 0; k < 64; k++) {
          // canonical layout: 8-element chunks along K, 448 rows (column half, digit, column)
          const size_t row = (size_t)(n / 32) * 224 + (size_t)(s - i) * 32 + (size_t)(n % 32);
          const size_t at = (size_t)(k / 8) * 448 * 8 + row * 8 + (size_t)(k % 8);
          sum += (int64_t)half_value(B[at]) * oz_digit(w[k], i);
        }
      if (s <= 4) worst[1] = std::max(worst[1], (double)std::llabs(sum));
      l[s] = (float)sum;   // exact up to weight 4; above, rounded at most a few times
    }
    const int64_t t = oz_sum(l);
    const int k2 = (int)E + eu - 1081;
    bool ok;
    const uint64_t bits = oz_round(t, k2, &ok);
    if (ok) std::memcpy(&out[n], &bits, 8);
    else out[n] = std::ldexp((double)t, k2);
    long double ref = 0;
    const int r = n / 2;
    for (int c = 0; c < 32; c++) {
      const long double a = u[2 * (32 * r + c)], b = u[2 * (32 * r + c) + 1];
      ref += (n & 1) ? b * x[2 * c] + a * x[2 * c + 1] : a * x[2 * c] - b * x[2 * c + 1];
    }
    if (norm > 0) worst[0] = std::max(worst[0], (double)(std::fabs((long double)out[n] - ref) / norm));
  }
  return 0;
}
