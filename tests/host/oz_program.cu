// Host interpreter of the exact tensor-core passes of complex128 programs (test
// only): the program the library builds for a circuit, every block's packed
// digits and parts applied to every row as the kernel does.
#include <cmath>
#include <cstring>
#include <vector>

#include "../../paper_2106_13995_gb300/csrc/oz_digits.cuh"
#include "../../paper_2106_13995_gb300/csrc/sv_internal.h"

using namespace sv;

static int half_int(uint16_t h) {
  const int e = (h >> 10) & 31, m = h & 1023;
  const double v = e ? std::ldexp(1024.0 + m, e - 25) : 0.0;
  return (int)((h & 0x8000) ? -v : v);
}

static void words(double v, uint32_t &hi, uint32_t &lo) {
  uint64_t b;
  std::memcpy(&b, &v, 8);
  hi = (uint32_t)(b >> 32);
  lo = (uint32_t)b;
}

// Applies the circuit to psi; returns the number of blocks on the tensor cores,
// 0 when the program has none (psi is left alone), -1 on an error, -2 when it
// has other passes as well.
extern "C" int oz_program(const sv_circuit *c, double *psi_) {
  sv_state s;
  s.n = c->n_qubits;
  s.dt = SV_C128;
  ProgramRef cp;
  Opts o;
  if (get_program(&s, c, nullptr, nullptr, &cp, &o) != SV_OK) return -1;
  int oz = 0;
  for (const TilePass &p : cp->prog.passes) oz += (p.flags & kPassOz) != 0;
  if (oz == 0) return 0;
  if (oz != (int)cp->prog.passes.size()) return -2;
  cd *psi = reinterpret_cast<cd *>(psi_);
  int blocks = 0;
  std::vector<int> B((size_t)kOzDigits * 64 * 64);   // digit j of (result n, input k)
  for (size_t pi = 0; pi < cp->prog.passes.size(); pi++) {
    const TilePass &p = cp->prog.passes[pi];
    for (int oi = 0; oi < p.nops; oi++, blocks++) {
      const TileOp &op = cp->prog.ops[cp->op0s[pi] + oi];
      const uint8_t *packed = cp->prog.mats.data() + 16 * (size_t)op.mat, *parts = packed + kOzOperandBytes;
      for (int j = 0; j < kOzDigits; j++)
        for (int n = 0; n < 64; n++)
          for (int k = 0; k < 64; k++) {
            // 8-element chunks along K, 448 rows (half of the results, digit, result)
            const size_t row = (size_t)(n / 32) * 224 + (size_t)j * 32 + n % 32;
            uint16_t h;
            std::memcpy(&h, packed + 2 * ((size_t)(k / 8) * 448 * 8 + row * 8 + k % 8), 2);
            B[((size_t)j * 64 + n) * 64 + k] = half_int(h);
          }
      uint64_t off[32], fixed = 0;
      for (int y = 0; y < 32; y++) {
        off[y] = 0;
        for (int j = 0; j < 5; j++) {
          const int t = op.t[j], q = t < p.L ? t : p.hi_pos[t - p.L];
          fixed |= 1ull << q;
          off[y] |= (uint64_t)((y >> j) & 1) << q;
        }
      }
      for (uint64_t base = 0; base < 1ull << p.n; base++) {
        if (base & fixed) continue;
        uint32_t E[32], hi[64], lo[64];
        for (uint32_t &e : E) e = 1;
        double x[64];
        for (int k = 0; k < 64; k++) {
          const cd v = psi[base | off[k / 2]];
          x[k] = (k & 1) ? v.imag() : v.real();
          words(x[k], hi[k], lo[k]);
          E[parts[k / 2]] = std::max(E[parts[k / 2]], oz_exponent(hi[k]));
        }
        int d[kOzDigits][64];
        for (int k = 0; k < 64; k++) {
          const uint64_t w = oz_fields(hi[k], lo[k], E[parts[k / 2]]);
          for (int i = 0; i < kOzDigits; i++) d[i][k] = oz_digit(w, i);
        }
        double out[64];
        for (int n = 0; n < 64; n++) {
          float l[kOzDigits];
          for (int w = 0; w < kOzDigits; w++) {
            int64_t sum = 0;
            for (int i = 0; i <= w; i++) {
              const int *b = &B[((size_t)(w - i) * 64 + n) * 64];
              int part = 0;   // 64 products of at most 2^16
              for (int k = 0; k < 64; k++) part += b[k] * d[i][k];
              sum += part;
            }
            l[w] = (float)sum;
          }
          const int64_t t = oz_sum(l);
          const int k2 = (int)E[parts[32 + n / 2]] + op.slot - 1081;
          bool ok;
          const uint64_t bits = oz_round(t, k2, &ok);
          if (ok) std::memcpy(&out[n], &bits, 8);
          else out[n] = std::ldexp((double)t, k2);
        }
        for (int y = 0; y < 32; y++) psi[base | off[y]] = cd(out[2 * y], out[2 * y + 1]);
      }
    }
  }
  return blocks;
}
