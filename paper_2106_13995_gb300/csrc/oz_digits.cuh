// FP64 numbers as signed 9-bit digits, and back: the arithmetic of the
// exact-product tensor-core blocks (k_tile_oz.cu), for the device and for the
// host that packs the matrices.
//
// A number v with |v| < 2^e is the integer q = trunc(v 2^(62 - e)), and
// q = sum_i d_i 2^(54 - 9 i), i = 0..6, with d_i in [-256, 256]: integers that
// FP16 holds exactly.  A product of two such digits is at most 2^16, and 64 x 4
// of them stay within the 24 bits an FP32 sum holds exactly, so a 64-term dot
// product splits into 7 x 7 digit products whose sums by weight i + j are
// exact in the tensor cores' FP32 accumulators (the splitting of Ozaki, Ogita,
// Oishi and Rump, Numerical Algorithms 59, 2012).  Weights i + j <= 6 are
// kept.  What is dropped is at most 2^-60 of 2^e times the matrix's 2^e a term:
// digits of random signs add up to about as much in a dot product, 64 terms of
// one sign to 2^-54.
#pragma once

#include <stdint.h>

#include <cmath>
#include <cstring>

namespace sv {

constexpr int kOzDigits = 7;
// sum of 256 * 2^(9 i), i < 7: added to q it makes every digit's field
// non-negative (field = digit + 256; the top one may reach 512)
constexpr uint64_t kOzBias = 256ull * (((1ull << 63) - 1) / 511);
static_assert(511ull * (((1ull << 63) - 1) / 511) == (1ull << 63) - 1, "2^63 - 1 is a multiple of 2^9 - 1");

// Biased exponent field of a double's high word (or of the largest of several
// high words without their signs), denormals as 1.
__host__ __device__ __forceinline__ uint32_t oz_exponent(uint32_t hi) {
  const uint32_t ex = (hi >> 20) & 0x7ffu;
  return ex ? ex : 1u;
}

// v (its two words) as biased digit fields, for a row whose largest exponent
// field is E >= v's: q + kOzBias with q = v 2^(62 - (E - 1022)), truncated.
__host__ __device__ __forceinline__ uint64_t oz_fields(uint32_t hi, uint32_t lo, uint32_t E) {
  const uint32_t ex = (hi >> 20) & 0x7ffu;
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32) | lo;
  const uint32_t d = E - (ex ? ex : 1u);
  const uint64_t q = (m << 9) >> (d < 63u ? d : 63u);
  const uint64_t s = (hi >> 31) ? ~0ull : 0ull;
  return ((q ^ s) - s) + kOzBias;
}

// Digit i of the fields.
__host__ __device__ __forceinline__ int oz_digit(uint64_t w, int i) {
  const uint32_t f = (uint32_t)(w >> (54 - 9 * i));
  return (int)(i == 0 ? f & 1023u : f & 511u) - 256;
}

// The sums by weight, as the tensor cores leave them, joined to an integer:
// T / 2^11 with T = sum_s l[s] 2^(54 - 9 s), |T| < 2^74.  The last two weights
// are joined in FP32 first (their sum is at most 2^22 quarters, rounded to a
// unit that is 2^-59 of a result of the row's size); l[0] 512 + l[1] fits 32
// bits, and the result 64, for the matrices oz_pack_matrix accepts.
__host__ __device__ __forceinline__ int64_t oz_sum(const float (&l)[kOzDigits]) {
#ifdef __CUDA_ARCH__
  const int c = __float2int_rn(fmaf(l[6], 0x1p-11f, l[5] * 0.25f));
#else
  const int c = (int)std::nearbyint(std::fma(l[6], 0x1p-11f, l[5] * 0.25f));
#endif
  const int u = (int)l[0] * 512 + (int)l[1];
  const int64_t v = (int64_t)u * 512 + (int)l[2];
  const int64_t w = (int64_t)(int)l[3] * 65536 + ((int64_t)(int)l[4] * 128 + c);
  return v * (1 << 25) + w;
}

// The bits of t 2^k rounded to nearest (ties away from zero), t != 0, in
// integers: the GB300's conversion from 64-bit integers runs at the FP64
// pipe's rate, and was half of the kernel's time.  *ok: the result is a normal
// number (else the bits are meaningless).
__host__ __device__ __forceinline__ uint64_t oz_round(int64_t t, int k, bool *ok) {
  const uint64_t s = (uint64_t)(t >> 63);
  uint64_t a = ((uint64_t)t ^ s) - s;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  a <<= lz & 63;                                        // bit 63 set
  const uint64_t m = (a >> 11) + ((a >> 10) & 1u);      // 53 bits, or 2^53
  const int e = 1086 - lz + k;                          // biased exponent of bit 63
  *ok = t != 0 && e >= 1 && e <= 2045;
  return (s & 0x8000000000000000ull) | (((uint64_t)(uint32_t)(e - 1) << 52) + m);
}

}  // namespace sv
