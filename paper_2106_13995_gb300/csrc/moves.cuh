// Permutation runs (k_moves.cu): descriptors and the index arithmetic that the
// kernel and its host emulation share.
#pragma once

#include <stdint.h>

namespace sv {

// A run of permutation gates is a list of multi-controlled X.  A thread follows
// 32 amplitudes at once: one 32-bit word ("plane") per index bit, and an X is
// one XOR of planes.
constexpr int kMoveThreads = 128;
constexpr int kMoveBits = 12;                 // amplitudes per CTA: 5 lane, 5 word and 2 warp bits
constexpr int kMovePlanes = 25;               // chunk bits (at most 22), all-ones, scratch, idle
constexpr uint32_t kMovePlaneBytes = kMoveThreads * 4;

// t ^= c1 & c2 (byte offsets of planes), or t = c1 & c2 with keep = 0, in CTAs
// whose known qubits (outside the chunk, or fixed for the CTA and never moved)
// read 1 at all of `gate`.
struct MoveOp {
  uint64_t gate;
  uint16_t t, c1, c2, keep;   // keep: 0xffff or 0
};
static_assert(sizeof(MoveOp) == 16, "MoveOp layout");
// Matrix-pool header (16-byte aligned) in front of the ops, which undo the run
// last gate first: they map an amplitude's place to where it came from.
struct MoveDesc {
  uint32_t nops;
  uint32_t pmask;             // chunk bits that have a plane
  uint8_t ord[32];            // chunk bit of lane bits 0-4, word bits 0-4, warp bits, CTA bits
  uint16_t plane[32];         // byte offset of a chunk bit's plane, 0xffff: none
  uint16_t ones, tmp, idle, pad;
};
static_assert(sizeof(MoveDesc) == 112, "MoveDesc layout");

// Word-bit patterns: bit w of word_pattern(k) is bit k of w.
__host__ __device__ constexpr uint32_t word_pattern(int k) {
  return k == 0 ? 0xAAAAAAAAu : k == 1 ? 0xCCCCCCCCu : k == 2 ? 0xF0F0F0F0u : k == 3 ? 0xFF00FF00u : 0xFFFF0000u;
}
// CTA or warp or lane bits of an index, by the order's chunk bits
__host__ __device__ __forceinline__ uint32_t move_deposit(uint32_t v, const uint8_t *ord, int from) {
  uint32_t r = 0;
  for (int k = 0; v >> k; k++) r |= ((v >> k) & 1u) << ord[from + k];
  return r;
}
// 32 x 32 bit transpose: bit k of r[w] becomes bit w of r[k] (halves, quarters,
// ... swapped across the diagonal).
template <int J> __host__ __device__ __forceinline__ void transpose_step(uint32_t (&r)[32], uint32_t m) {
#pragma unroll
  for (int k = 0; k < 32; k++)
    if (!(k & J)) {
      const uint32_t t = ((r[k] >> J) ^ r[k | J]) & m;
      r[k | J] ^= t;
      r[k] ^= t << J;
    }
}
__host__ __device__ __forceinline__ void transpose32(uint32_t (&r)[32]) {
  transpose_step<16>(r, 0x0000FFFFu);
  transpose_step<8>(r, 0x00FF00FFu);
  transpose_step<4>(r, 0x0F0F0F0Fu);
  transpose_step<2>(r, 0x33333333u);
  transpose_step<1>(r, 0x55555555u);
}

}  // namespace sv
