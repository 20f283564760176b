// K14: tile passes of dense 5-qubit blocks of complex128 states on the tensor
// cores, exactly (12-qubit tiles).
//
// The GB300 multiplies FP64 at two FMAs a clock and SM, and a fused 3-qubit
// block needs 32 of them per amplitude.  Here a block is the GEMM of K9 (M =
// 128 groups, N = K = 64, the real embedding of U) on digits: every FP64
// number becomes seven signed 9-bit integers (oz_digits.cuh) relative to the
// largest number of its group's part (oz_parts), the 28 products of digits i, j with i + j <= 6
// run as FP16 MMAs whose FP32 sums are exact integers, and the seven sums per
// result are joined in 64-bit integers and rounded to FP64 once.  No FP64
// arithmetic is left but one integer conversion per number.
//
// One persistent CTA per SM: 512 threads, four to a row (TMEM lane).  Per
// block: every thread gathers 8 amplitudes of its row from the tile in shared
// memory, finds the parts' exponents with the row's other threads, and stores
// the digits as FP16 A operands in TMEM (224 columns); one thread issues the
// MMAs of the first 32 result columns (7 x 32 TMEM columns of sums); the
// threads read those sums, the MMAs of the other 32 columns start, and the
// first half is joined and scattered while they run.  The B operands (56 KB a
// block) are copied from L2 into two buffers in turn.
//
// An MMA of M = 128 and K = 16 with A in TMEM takes about 50 clocks up to N =
// 64, so digit i of A meets all its digits of B in one of N = 32 (7 - i): 56
// MMAs per tile and block.  One MMA of N = 32 per digit product (224) took 0.42
// of the time: 1.78 ms against 1.24 for 33 blocks of 21 qubits.
//
// Bound (21 qubits, 9.3 us per tile and block): the chain gather - digits - MMA
// - join of one tile; without the join 0.28 less, with a seventh of the MMAs
// 0.13 less.  A 23-qubit grid circuit of 20 cycles: 24.1 ms in FP64 arithmetic,
// 4.5 ms here (4.3 with one exponent for all of a row, which lost the low bits of
// small amplitudes next to large ones that their block does not mix).
//
// Every wait is bounded, as in K9.
#include <algorithm>
#include <cstring>
#include <vector>

#include <cuda_fp16.h>

#include "oz_digits.cuh"
#include "sv_device.cuh"
#include "sv_internal.h"

namespace sv {

constexpr int kOzThreads = 512;
constexpr uint32_t kOzTileBytes = (1u << kTcTileM) * 16;     // 64 KB
constexpr uint32_t kOzBRows = kOzDigits * 64;                 // of B: half of the columns, digit, 32 columns
constexpr uint32_t kOzBBytes = kOzBRows * 64 * 2;             // 56 KB
// largest high words of the members (or of the threads' shares) and exponents
// of the parts, 32 x 128 each
constexpr uint32_t kOzSmB = kOzTileBytes, kOzSmHi = kOzSmB + 2 * kOzBBytes, kOzSmExp = kOzSmHi + 32 * 128 * 4;
constexpr uint32_t kOzSmBar = kOzSmExp + 32 * 128 * 4;
constexpr uint32_t kOzSmem = kOzSmBar + 8 * 3 + 8;
static_assert(kOzSmem <= 227u * 1024u, "shared memory of a CTA");
constexpr uint32_t kOzTmemCols = 512, kOzTmemD = kOzDigits * 32;   // A digits, then the sums
static_assert(2 * kOzDigits * 32 <= (int)kOzTmemCols, "TMEM columns");
constexpr uint32_t kOzSpin = 1u << 22;

// Per block: member offsets and row-bit offsets in the tile, and the exponent
// of the matrix.
struct OzTable {
  uint32_t soff[kOzMaxBlocks][32];
  uint32_t rbit[kOzMaxBlocks][7];
  int32_t eu[kOzMaxBlocks];
  uint32_t mat[kOzMaxBlocks];   // 16-byte index of the packed operand in the pool
  // parts of the block: their number, each one's input members as a mask, and
  // the part of every input and output member
  uint32_t nparts[kOzMaxBlocks];
  uint32_t mask[kOzMaxBlocks][32];
  uint8_t in[kOzMaxBlocks][32], out[kOzMaxBlocks][32];
};
static_assert(kOzBBytes == kOzOperandBytes, "operand size");

// byte offset of tile amplitude l (linear over GF(2)); see tcp_row_positions
// for how lanes are kept apart
__host__ __device__ constexpr uint32_t oz_slot(uint32_t l) { return (l ^ (((l >> 3) ^ (l >> 6) ^ (l >> 9)) & 7u)) * 16u; }

__device__ __forceinline__ void oz_tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void oz_tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// D (TMEM) += A (TMEM) x B (shared memory), FP16 inputs, FP32 accumulation
__device__ __forceinline__ void oz_mma(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(bdesc), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void oz_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// (one thread) result columns 32 h .. 32 h + 31: every digit product of weight
// at most 6 into the sum of its weight.  Digit i of A meets digits 0 .. 6 - i
// of B in one MMA: their operands follow each other by 32 rows, as the sums of
// weight i and up do by 32 columns.
__device__ __forceinline__ void oz_issue(uint32_t tmem, uint32_t bs, int h) {
  // descriptors differ in their address field alone (16-byte units)
  const uint64_t b0 = smem_desc(bs + (uint32_t)h * (kOzBRows / 2) * 16, kOzBRows * 16, 128);
#pragma unroll
  for (uint32_t k = 0; k < 4; k++)
#pragma unroll
    for (uint32_t i = 0; i < kOzDigits; i++)
      oz_mma(tmem + kOzTmemD + 32 * i, tmem + 32 * i + 8 * k, b0 + (uint64_t)(2 * k * kOzBRows),
             instr_desc(0u, 128, (kOzDigits - i) * 32), (i > 0 || k > 0) ? 1u : 0u);   // FP16 A and B, FP32 D
}

// A denormal, infinite or zero result.  Out of line: inlined, its FP64
// operations run for every result, selected away afterwards.
__device__ __noinline__ double oz_rare(int64_t t, int k) { return t == 0 ? 0.0 : ldexp(__ll2double_rn(t), k); }

// A result from its seven sums.
__device__ __forceinline__ double oz_join(const uint32_t (&v)[kOzDigits], int k, bool bad) {
  float l[kOzDigits];
#pragma unroll
  for (int s = 0; s < kOzDigits; s++) l[s] = __uint_as_float(v[s]);
  const int64_t t = oz_sum(l);
  bool ok;
  const uint64_t bits = oz_round(t, k, &ok);
  double d = __longlong_as_double((long long)bits);
  if (!ok) d = oz_rare(t, k);
  return bad ? __hiloint2double(0x7ff80000, 0) : d;
}

__global__ void __launch_bounds__(kOzThreads, 1)
    k_tile_oz(const __grid_constant__ TilePass P, const __grid_constant__ OzTable T) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint64_t s_trip[8];
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar_mma = sbase + kOzSmBar, bar_b = bar_mma + 8;
  uint32_t *slot = reinterpret_cast<uint32_t *>(smem + kOzSmBar + 24);
  uint32_t *shi = reinterpret_cast<uint32_t *>(smem + kOzSmHi), *sexp = reinterpret_cast<uint32_t *>(smem + kOzSmExp);
  const uint32_t tid = threadIdx.x, row = tid & 127u, g = tid >> 7;
  const int nb = P.nops;
  const uint32_t segmask = (1u << P.L) - 1;
  if (tid == 0) {
    for (int i = 0; i < 3; i++) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar_mma + 8 * i));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (tid < 8) {
    const uint32_t lt = tid * kOzThreads;
    uint64_t o = lt & segmask;
    for (uint32_t x = lt >> P.L; x; x &= x - 1) o |= 1ull << P.hi_pos[__ffs(x) - 1];
    s_trip[tid] = o;
  }
  if (tid < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot)),
                 "r"(kOzTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot, lane = (row & ~31u) << 16;
  const uint64_t ntiles = 1ull << (P.n - P.m);
  // blocks this CTA runs, and the copy of block c's operand into buffer c & 1
  const uint64_t mine = blockIdx.x < ntiles ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  const uint64_t total = mine * (uint64_t)nb;
  auto copy_b = [&](uint64_t c) {   // (thread 0)
    const uint32_t b = bar_b + 8 * (uint32_t)(c & 1);
    const char *src = static_cast<const char *>(P.mats) + 16 * (size_t)T.mat[c % (uint64_t)nb];
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(b), "r"(kOzBBytes) : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            sbase + kOzSmB + (uint32_t)(c & 1) * kOzBBytes),
        "l"(src), "r"(kOzBBytes), "r"(b)
        : "memory");
  };
  uint64_t copied = 0, c = 0;
  if (tid == 0)
    for (; copied < 2 && copied < total; copied++) copy_b(copied);
  pass_wait();
  uint64_t thr = tid & segmask;
  for (uint32_t x = tid >> P.L; x; x &= x - 1) thr |= 1ull << P.hi_pos[__ffs(x) - 1];
  double2 *amps = reinterpret_cast<double2 *>(P.v0);
  uint32_t phase = 0;       // of bar_mma
  bool pending = false;     // (thread 0) MMAs committed but not observed
  bool failed = false;
  for (uint64_t t = blockIdx.x; t < ntiles && !failed; t += gridDim.x) {
    uint64_t base = 0;
    for (uint64_t x = t; x; x &= x - 1) base |= 1ull << P.out_pos[__ffsll((long long)x) - 1];
#pragma unroll
    for (uint32_t i = 0; i < 8; i++)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sbase + oz_slot(tid + i * kOzThreads)),
                   "l"(amps + (base | thr | s_trip[i]))
                   : "memory");
    if (t + gridDim.x < ntiles) {   // the next tile towards L2
      uint64_t nxt = 0;
      for (uint64_t x = t + gridDim.x; x; x &= x - 1) nxt |= 1ull << P.out_pos[__ffsll((long long)x) - 1];
#pragma unroll
      for (uint32_t i = 0; i < 8; i++)
        asm volatile("prefetch.global.L2 [%0];\n" ::"l"(amps + (nxt | thr | s_trip[i])));
    }
    cp_async_wait_all();
    __syncthreads();
    for (int bi = 0; bi < nb; bi++, c++) {
      uint32_t s0 = 0;
#pragma unroll
      for (int b = 0; b < 7; b++) s0 ^= ((row >> b) & 1u) ? T.rbit[bi][b] : 0u;
      // gather, and the exponents of the row's parts
      double2 x[8];
      uint32_t hi[8];   // largest high word without its sign
#pragma unroll
      for (int j = 0; j < 8; j++) {
        x[j] = *reinterpret_cast<const double2 *>(smem + (s0 ^ T.soff[bi][8 * g + j]));
        hi[j] = max((uint32_t)__double2hiint(x[j].x) & 0x7fffffffu, (uint32_t)__double2hiint(x[j].y) & 0x7fffffffu);
      }
      const uint32_t np = T.nparts[bi];
      uint32_t E = 0;   // of the row, where the block is one part
      if (np == 1) {
#pragma unroll
        for (int j = 0; j < 8; j++) E = max(E, hi[j]);
        shi[g * 128 + row] = E;
        __syncthreads();
        E = oz_exponent(max(max(shi[row], shi[128 + row]), max(shi[256 + row], shi[384 + row])));
      } else {
#pragma unroll
        for (int j = 0; j < 8; j++) shi[(8 * g + j) * 128 + row] = hi[j];
        __syncthreads();
        for (uint32_t p = g; p < np; p += 4) {
          uint32_t e = 0;
          for (uint32_t m = T.mask[bi][p]; m; m &= m - 1) e = max(e, shi[(__ffs(m) - 1) * 128 + row]);
          sexp[p * 128 + row] = oz_exponent(e);
        }
        __syncthreads();
      }
      // digits: fields of (re, im) side by side as FP16 1024 + field, less 1280
      uint64_t wr[8], wi[8];
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const uint32_t e = np == 1 ? E : sexp[T.in[bi][8 * g + j] * 128 + row];
        wr[j] = oz_fields((uint32_t)__double2hiint(x[j].x), (uint32_t)__double2loint(x[j].x), e);
        wi[j] = oz_fields((uint32_t)__double2hiint(x[j].y), (uint32_t)__double2loint(x[j].y), e);
      }
#pragma unroll
      for (int i = 0; i < kOzDigits; i++) {
        uint32_t a[8];
        const uint32_t mask = i == 0 ? 0x03ff03ffu : 0x01ff01ffu;
        const int sh = 54 - 9 * i;
#pragma unroll
        for (int j = 0; j < 8; j++) {
          // re's field to bit 0, im's to bit 16
          const uint32_t re = (uint32_t)(wr[j] >> sh);
          const uint32_t im = sh >= 16 ? (uint32_t)(wi[j] >> (sh >= 16 ? sh - 16 : 0)) : (uint32_t)wi[j] << (sh < 16 ? 16 - sh : 0);
          const uint32_t f = (__byte_perm(re, im, 0x7610) & mask) | 0x64006400u;
          const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&f), __halves2half2(__ushort_as_half(0x6500), __ushort_as_half(0x6500)));
          a[j] = *reinterpret_cast<const uint32_t *>(&h);
        }
        oz_tmem_st8(tmem + lane + 32 * i + 8 * g, a);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
      tc_fence_before();
      __syncthreads();
      const uint32_t bs = sbase + kOzSmB + (uint32_t)(c & 1) * kOzBBytes;
      bool ok = true;
      if (tid == 0) {
        tc_fence_after();
        ok = mbar_wait(bar_b + 8 * (uint32_t)(c & 1), (uint32_t)(c >> 1) & 1u, kOzSpin);
        if (ok) {
          oz_issue(tmem, bs, 0);
          oz_commit(bar_mma);
          pending = true;
        }
      }
      // (if the operand never landed nothing was committed, and the wait below
      // runs out)
#pragma unroll
      for (int h = 0; h < 2; h++) {
        ok = ok && mbar_wait(bar_mma, phase, kOzSpin);
        phase ^= 1u;
        if (ok && tid == 0) pending = false;
        tc_fence_after();
        uint32_t r[kOzDigits][8];
#pragma unroll
        for (int s = 0; s < kOzDigits; s++) oz_tmem_ld8(tmem + lane + kOzTmemD + 32 * s + 8 * g, r[s]);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        tc_fence_before();
        if (__syncthreads_or(!ok)) {
          failed = true;
          break;
        }
        if (tid == 0) {
          tc_fence_after();
          if (h == 0) {
            oz_issue(tmem, bs, 1);
            oz_commit(bar_mma);
            pending = true;
          } else if (copied < total) {
            copy_b(copied++);   // both halves are done with this buffer
          }
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
          double2 o;
          uint32_t v[kOzDigits];
          const uint32_t e = np == 1 ? E : sexp[T.out[bi][16 * h + 4 * g + j] * 128 + row];
          const int k = (int)e + T.eu[bi] - 1081;
          const bool bad = e == 0x7ffu;
#pragma unroll
          for (int s = 0; s < kOzDigits; s++) v[s] = r[s][2 * j];
          o.x = oz_join(v, k, bad);
#pragma unroll
          for (int s = 0; s < kOzDigits; s++) v[s] = r[s][2 * j + 1];
          o.y = oz_join(v, k, bad);
          *reinterpret_cast<double2 *>(smem + (s0 ^ T.soff[bi][16 * h + 4 * g + j])) = o;
        }
      }
      if (failed) break;
      __syncthreads();
    }
    if (failed) break;
    if (t + gridDim.x >= ntiles) pass_start();
#pragma unroll
    for (uint32_t i = 0; i < 8; i++)
      __stcs(reinterpret_cast<int4 *>(amps + (base | thr | s_trip[i])),
             *reinterpret_cast<const int4 *>(smem + oz_slot(tid + i * kOzThreads)));
    __syncthreads();
  }
  // no copy or MMA may outlive the CTA
  if (failed && tid == 0) atomicExch(P.err, 1u);
  if (tid == 0) {
    if (pending) mbar_wait(bar_mma, phase, kOzSpin);
    for (uint64_t i = copied >= 2 ? copied - 2 : 0; i < copied; i++)
      mbar_wait(bar_b + 8 * (uint32_t)(i & 1), (uint32_t)(i >> 1) & 1u, kOzSpin);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(*slot), "r"(kOzTmemCols));
}

// ---------------------------------------------------------------------------
// host: operands
// ---------------------------------------------------------------------------
static std::pair<uint32_t, uint32_t> oz_words(double v) {
  uint64_t b;
  std::memcpy(&b, &v, 8);
  return {(uint32_t)(b >> 32), (uint32_t)b};
}

// U (32 x 32) as FP16 digits of its real embedding in the canonical no-swizzle
// K-major layout: row 224 h + 32 i + c is digit i of result column 32 h + c; eu: |entries| < 2^eu.  False
// when a sum of weight at most 4 could pass 2^24 for some input (row sums of
// the digits' magnitudes; the weights beyond may: an FP32 rounding there is
// 2^-57 of a result), when the first weight's could pass 15/16 of 2^20 (the
// joined integer is T / 2^11, so 64 bits hold 2^20 of them), or an entry is not
// finite.  A matrix with a row sum of 15 largest entries or more takes its
// digits against 2 or 4 times the largest entry: the row's norm is then at
// least 2 or 4 of those (an eighth of the sum of its 64 numbers), so an error
// relative to the norm stays what it is.
static bool oz_pack_digits(const std::vector<cd> &U, std::vector<uint16_t> &out, uint32_t E);
bool oz_pack_matrix(const std::vector<cd> &U, std::vector<uint16_t> &out, int &eu) {
  uint32_t E = 1;
  for (const cd &u : U)
    for (double v : {u.real(), u.imag()}) E = std::max(E, oz_exponent(oz_words(v).first));
  if (E >= 0x7fd) return false;
  double sum = 0;
  for (int r = 0; r < 32; r++) {
    double row = 0;
    for (int q = 0; q < 32; q++) row += std::fabs(U[(size_t)r * 32 + q].real()) + std::fabs(U[(size_t)r * 32 + q].imag());
    sum = std::max(sum, std::ldexp(row, 1022 - (int)E));
  }
  for (uint32_t up = sum > 30 ? 2 : sum > 15 ? 1 : 0; up < 3; up++)
    if (oz_pack_digits(U, out, E + up)) {
      eu = (int)(E + up) - 1022;
      return true;
    }
  return false;
}

static bool oz_pack_digits(const std::vector<cd> &U, std::vector<uint16_t> &out, uint32_t E) {
  // FP16 bits of the integers -256..256
  struct Halves {
    uint16_t of[513];
    Halves() {
      for (int d = -256; d <= 256; d++) {
        const uint32_t a = (uint32_t)(d < 0 ? -d : d);
        const int e = a ? 31 - __builtin_clz(a) : 0;
        of[d + 256] = a ? (uint16_t)((d < 0 ? 0x8000 : 0) | ((15 + e) << 10) | ((a << (10 - e)) & 0x3ffu)) : 0;
      }
    }
  };
  static const Halves halves;
  out.assign((size_t)kOzDigits * 64 * 64, 0);
  std::vector<uint32_t> mag((size_t)32 * kOzDigits, 0);   // digit magnitudes, summed along a row
  for (int r = 0; r < 32; r++)
    for (int q = 0; q < 32; q++)
      for (int part = 0; part < 2; part++) {
        const double v = part ? U[(size_t)r * 32 + q].imag() : U[(size_t)r * 32 + q].real();
        if (v == 0) continue;   // all digits 0
        const auto [hi, lo] = oz_words(v);
        const uint64_t w = oz_fields(hi, lo, E);
        // Re at (2r, 2q) and (2r + 1, 2q + 1); Im at (2r + 1, 2q), -Im at (2r, 2q + 1)
        auto at = [](int n, int k) {
          return (size_t)(cm_offset((uint32_t)(n / 32) * (kOzBRows / 2) + (uint32_t)(n % 32), (uint32_t)k / 8, kOzBRows) / 2) +
                 (size_t)(k % 8);
        };
        const size_t at0 = at(2 * r + part, 2 * q), at1 = at(2 * r + 1 - part, 2 * q + 1);
        for (int i = 0; i < kOzDigits; i++) {
          const int d = oz_digit(w, i);
          mag[(size_t)r * kOzDigits + i] += (uint32_t)(d < 0 ? -d : d);
          out[at0 + (size_t)i * 32 * 8] = halves.of[256 + d];
          out[at1 + (size_t)i * 32 * 8] = halves.of[256 + (part ? -d : d)];
        }
      }
  for (int r = 0; r < 32; r++) {
    uint64_t sum = 0;
    for (int i = 0; i < 5; i++) {
      sum += mag[(size_t)r * kOzDigits + i];
      if (sum * 256 > (i == 0 ? 15u << 16 : 1u << 24)) return false;
    }
  }
  return true;
}

// The parts of a block: inputs and outputs that its gates connect (mag: the
// product of the gates' entry magnitudes), labelled 0, 1, ...; in[y] and out[y]
// are the labels of member y.  A control, an idle or padding qubit, a diagonal
// or a permuted one splits the members, and digits are relative to the largest
// number of a part.  FP64 arithmetic leaves a result within rounding of
// sum_y mag[r][y] |x_y|; the digits add about 2^-60 of the powers of two above
// the part's largest number and above the matrix's entries (2^eu).  So a block
// qualifies where every entry of mag within a part is at least 2^-6 2^eu: the
// digits' share is then at most about one FP64 rounding of that sum, whatever
// the amplitudes are.  Others (a rotation by a small angle next to a large
// amplitude) keep FP64 arithmetic.
bool oz_parts(const std::vector<double> &mag, int eu, uint8_t *in, uint8_t *out) {
  double least = HUGE_VAL;
  int root[64];   // inputs 0..31, outputs 32..63
  for (int x = 0; x < 64; x++) root[x] = x;
  auto find = [&](int x) {
    while (root[x] != x) x = root[x] = root[root[x]];
    return x;
  };
  int entries = 0;
  for (int r = 0; r < 32; r++)
    for (int y = 0; y < 32; y++) {
      const double m = mag[(size_t)r * 32 + y];
      if (m == 0) continue;
      if (!(m > 0)) return false;
      least = std::min(least, m);
      entries++;
      root[find(32 + r)] = find(y);
    }
  if (!(least >= std::ldexp(1.0, eu - 6))) return false;
  int label[64], n = 0, ins[32] = {}, outs[32] = {};
  std::fill(label, label + 64, -1);
  for (int y = 0; y < 32; y++) {
    const int f = find(y);
    if (label[f] < 0) label[f] = n++;
    in[y] = (uint8_t)label[f];
    ins[in[y]]++;
  }
  for (int r = 0; r < 32; r++) {
    const int f = find(32 + r);
    if (label[f] < 0) return false;   // a row of zeros
    out[r] = (uint8_t)label[f];
    outs[out[r]]++;
  }
  for (int p = 0; p < n; p++) entries -= ins[p] * outs[p];
  return entries == 0;   // every input of a part reaches every output of it
}

// Row bits of a block: the first three lane bits take tile positions of
// different bank classes ({0,3,6,9}, {1,4,7,10}, {2,5,8,11}: 8 lanes of a
// 16-byte access then reach 8 banks), the others follow in order.
static void oz_rows(const TileOp &op, int *rows) {
  uint32_t used = 0;
  for (int j = 0; j < 5; j++) used |= 1u << op.t[j];
  int k = 0;
  for (int cls = 0; cls < 3; cls++)
    for (int p = cls; p < kTcTileM; p += 3)
      if (!((used >> p) & 1u)) {
        rows[k++] = p;
        used |= 1u << p;
        break;
      }
  for (int p = 0; p < kTcTileM && k < 7; p++)
    if (!((used >> p) & 1u)) rows[k++] = p;
}

sv_status launch_tile_oz(sv_state *s, const TilePass &p, const HostPass &host, cudaStream_t stream) {
  if (s->dt != SV_C128 || p.m != kTcTileM || p.nops < 1 || p.nops > kOzMaxBlocks)
    return set_error(SV_EINVAL, "internal: not an exact tensor-core pass");
  SV_TRY(func_attr_once((const void *)k_tile_oz, s->device, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmem));
  OzTable T;
  std::memset(&T, 0, sizeof(T));
  for (int i = 0; i < p.nops; i++) {
    const TileOp &op = host.ops[i];
    for (int y = 0; y < 32; y++) {
      uint32_t l = 0;
      for (int j = 0; j < 5; j++) l |= (uint32_t)((y >> j) & 1) << op.t[j];
      T.soff[i][y] = oz_slot(l);
    }
    int rows[7];
    oz_rows(op, rows);
    for (int b = 0; b < 7; b++) T.rbit[i][b] = oz_slot(1u << rows[b]);
    T.eu[i] = op.slot;
    T.mat[i] = op.mat;
    const uint8_t *parts = host.mats + 16 * (size_t)op.mat + kOzOperandBytes;
    for (int y = 0; y < 32; y++) {
      T.in[i][y] = parts[y];
      T.out[i][y] = parts[32 + y];
      T.mask[i][parts[y]] |= 1u << y;
      T.nparts[i] = std::max(T.nparts[i], parts[y] + 1u);
    }
  }
  const uint64_t ntiles = 1ull << (p.n - p.m);
  const int grid = (int)std::min<uint64_t>(ntiles, (uint64_t)s->sm_count);
  SV_CUDA(launch_early(k_tile_oz, dim3((unsigned)grid), kOzThreads, kOzSmem, stream, p, T));
  g_launches++;
  return SV_OK;
}

}  // namespace sv
