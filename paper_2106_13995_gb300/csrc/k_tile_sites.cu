// K13: passes of gradient programs made of TOP_SITES ops (complex64; one or
// two vectors per tile, all parameter sets of a batch in grid.y).
//
// Bound: issue slots (20 qubits, 8 sets, reverse pass of 5 ops: 150 us, 2.3
// instructions a clock, 18% of HBM; 225 us as one op per gate and CNOT).
// 12-qubit tiles, three CTAs of 256 threads per SM.  64 gradients of the
// 20-qubit, 10-layer ansatz: 109.8 -> 40.8 ms; one of 16 qubits and 6 layers
// 1.41 -> 0.48 ms.
#include <algorithm>
#include <cstring>

#include "tile_ops.cuh"

namespace sv {

constexpr int kSitesThreads = 256;
constexpr uint32_t kSitesEntry = 14;     // 16-byte words per op: op, descriptor, three matrices

// A step of a gradient program on three tile qubits (complex64): each thread
// holds the 8 amplitudes of a group -- of psi and, in the reverse sweep, of
// lambda -- in registers, loaded through the moves before and stored through
// the moves after; between them every target with a site takes its probes
// (Im <lambda | G | psi> for G = X, Y, Z in its mask; all generators of a run
// of gates on one qubit follow from these) and its 1-qubit matrix on both
// vectors.  One shared-memory read and write per amplitude for up to three
// runs and the permutations around them, where each gate and permutation was
// a sweep of its own.  The two vectors' components are packed in pairs, so a
// matrix costs 8 packed FMAs per amplitude of both.
template <bool TWO>
__device__ __forceinline__ void sites_op(uint32_t vs0, uint32_t vs1, int m, const uint4 *e, float *red) {
  // the entry: op, descriptor, matrices (shared memory, the same for all threads)
  TileOp op;
  {
    const uint4 o[2] = {e[0], e[1]};
    memcpy(&op, o, sizeof(op));
  }
  const uint4 mq = e[6], sq = e[7];
  // (member offsets are read where they are used: 16 registers)
  const volatile uint32_t *ld = reinterpret_cast<const volatile uint32_t *>(e + 2), *st = ld + 8;
  const int mat[3] = {(int)mq.x, (int)mq.y, (int)mq.z};
  const uint32_t comps = sq.w;
  const uint32_t tid = threadIdx.x, T = blockDim.x;
  const uint32_t fixed = (1u << op.t[0]) | (1u << op.t[1]) | (1u << op.t[2]);
  const uint32_t ngroups = 1u << (m - 3);
  const uint32_t ntrips = tid < ngroups ? (ngroups > T ? ngroups / T : 1u) : 0u;
  const uint32_t sthr = swb<float>(thread_l(tid, op));
  const TripMap tm = trip_map(T, fixed);
  float px[3] = {0, 0, 0}, py[3] = {0, 0, 0}, pz[3] = {0, 0, 0};
  for (uint32_t c = 0; c < ntrips; c++) {
    const uint32_t s = sthr ^ swb<float>(trip_l(c, tm));
    uint64_t x[8], y[8];   // (psi, lambda) real and imaginary parts; psi alone: x holds (re, im)
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const uint32_t at = s ^ ld[i];
      const float2 a = lds_c(vs0 + at, (const float2 *)nullptr);
      if constexpr (TWO) {
        const float2 b = lds_c(vs1 + at, (const float2 *)nullptr);
        x[i] = pk2(a.x, b.x);
        y[i] = pk2(a.y, b.y);
      } else {
        x[i] = pk2(a.x, a.y);
      }
    }
#pragma unroll
    for (int J = 0; J < 3; J++) {
      if (mat[J] < 0) continue;
      if constexpr (TWO) {
        if ((comps >> (4 * J)) & 15u) {
#pragma unroll
          for (int i = 0; i < 8; i++)
            if (!((i >> J) & 1)) {
              const int k = i | (1 << J);
              const float2 x0 = upk2(x[i]), y0 = upk2(y[i]), x1 = upk2(x[k]), y1 = upk2(y[k]);
              const float2 a0 = make_float2(x0.x, y0.x), b0 = make_float2(x0.y, y0.y);
              const float2 a1 = make_float2(x1.x, y1.x), b1 = make_float2(x1.y, y1.y);
              // Im <b | Z a>, Im <b | X a>, and Im <b | Y a> = Re(conj(b1) a0 - conj(b0) a1)
              pz[J] = fmaf(b0.x, a0.y, fmaf(-b0.y, a0.x, fmaf(b1.y, a1.x, fmaf(-b1.x, a1.y, pz[J]))));
              px[J] = fmaf(b0.x, a1.y, fmaf(-b0.y, a1.x, fmaf(b1.x, a0.y, fmaf(-b1.y, a0.x, px[J]))));
              py[J] = fmaf(b1.x, a0.x, fmaf(b1.y, a0.y, fmaf(-b0.x, a1.x, fmaf(-b0.y, a1.y, py[J]))));
            }
        }
      }
      // row pairs (Re U00, Re U10, Im U00, Im U10), then column 1
      const uint4 q0 = e[8 + 2 * J], q1 = e[9 + 2 * J];
      const float2 u00 = make_float2(__uint_as_float(q0.x), __uint_as_float(q0.z));
      const float2 u10 = make_float2(__uint_as_float(q0.y), __uint_as_float(q0.w));
      const float2 u01 = make_float2(__uint_as_float(q1.x), __uint_as_float(q1.z));
      const float2 u11 = make_float2(__uint_as_float(q1.y), __uint_as_float(q1.w));
#pragma unroll
      for (int i = 0; i < 8; i++)
        if (!((i >> J) & 1)) {
          const int k = i | (1 << J);
          if constexpr (TWO) {
            const uint64_t ax = x[i], ay = y[i], bx = x[k], by = y[k];
            const auto c2 = [](float v) { return pk2(v, v); };
            x[i] = fma2(c2(u00.x), ax, fma2(c2(-u00.y), ay, fma2(c2(u01.x), bx, fma2(c2(-u01.y), by, 0ull))));
            y[i] = fma2(c2(u00.x), ay, fma2(c2(u00.y), ax, fma2(c2(u01.x), by, fma2(c2(u01.y), bx, 0ull))));
            x[k] = fma2(c2(u10.x), ax, fma2(c2(-u10.y), ay, fma2(c2(u11.x), bx, fma2(c2(-u11.y), by, 0ull))));
            y[k] = fma2(c2(u10.x), ay, fma2(c2(u10.y), ax, fma2(c2(u11.x), by, fma2(c2(u11.y), bx, 0ull))));
          } else {
            const float2 a = upk2(x[i]), b = upk2(x[k]);
            const float2 p = cfma(u01, b, cmul(u00, a)), q = cfma(u11, b, cmul(u10, a));
            x[i] = pk2(p.x, p.y);
            x[k] = pk2(q.x, q.y);
          }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const uint32_t at = s ^ st[i];
      const float2 xv = upk2(x[i]);
      if constexpr (TWO) {
        const float2 yv = upk2(y[i]);
        sts_c(vs0 + at, make_float2(xv.x, yv.x));
        sts_c(vs1 + at, make_float2(xv.y, yv.y));
      } else {
        sts_c(vs0 + at, xv);
      }
    }
  }
  if constexpr (TWO) {
    // the warp's sums; flush_probes adds the warps' after the next barrier
#pragma unroll
    for (int J = 0; J < 3; J++) {
      const uint32_t cm = (comps >> (4 * J)) & 7u;
#pragma unroll
      for (int g = 0; g < 3; g++)
        if ((cm >> g) & 1u) {
          const float p = warp_sum(g == 0 ? px[J] : g == 1 ? py[J] : pz[J]);
          if ((tid & 31) == 0) red[(3 * J + g) * (kSitesThreads / 32) + (tid >> 5)] = p;
        }
    }
  }
}

// One FP64 atomic per probe and tile: thread 3 J + g adds the warps' sums of
// target J's component g (an atomic per warp was half of the kernel's time:
// all tiles of a set add to the same few addresses).
__device__ __forceinline__ void flush_probes(const uint4 *e, const float *red, double *__restrict__ acc) {
  const uint32_t t = threadIdx.x;
  if (t >= 9) return;
  const uint4 sq = e[7];
  const uint32_t J = t / 3, g = t % 3, cm = (sq.w >> (4 * J)) & 7u;
  if (!((cm >> g) & 1u)) return;
  double p = 0;
  for (uint32_t w = 0; w < (blockDim.x + 31) / 32; w++) p += (double)red[t * (kSitesThreads / 32) + w];
  const int slot = J == 0 ? (int)sq.x : J == 1 ? (int)sq.y : (int)sq.z;
  atomicAdd(acc + slot + __popc(cm & ((1u << g) - 1)), p);
}

template <bool TWO>
__global__ void __launch_bounds__(kSitesThreads, 3) k_tile_sites(const __grid_constant__ TilePass P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float red[2][9 * (kSitesThreads / 32)];   // the warps' probe sums of an op and of the one before
  const uint32_t TS = 1u << P.m, T = blockDim.x, nunits = TS / 2;
  float2 *g0 = reinterpret_cast<float2 *>(P.tbl0 ? P.tbl0[blockIdx.y] : P.v0);
  float2 *g1 = TWO ? reinterpret_cast<float2 *>(P.tbl1 ? P.tbl1[blockIdx.y] : P.v1) : nullptr;
  const uint32_t vs0 = smem_u32(smem_raw), vs1 = vs0 + TS * (uint32_t)sizeof(float2);
  uint4 *ent = reinterpret_cast<uint4 *>(smem_raw + (size_t)(TWO ? 2 : 1) * TS * sizeof(float2));
  const float2 *pm = reinterpret_cast<const float2 *>(P.pmats) + (size_t)blockIdx.y * P.pmats_stride;
  double *acc = P.acc ? P.acc + (size_t)blockIdx.y * P.acc_stride : nullptr;
  const uint64_t base = tile_base(P, blockIdx.x);
  const uint32_t segmask = (1u << P.L) - 1;
  const uint32_t lthr = threadIdx.x * 2;
  const uint64_t gthr = base | (lthr & segmask) | spread_hi(P, lthr & ~segmask);
  auto goff = [&](uint32_t i) -> uint64_t {
    const uint32_t lt = i * T * 2;
    return gthr | (lt & segmask) | spread_hi(P, lt & ~segmask);
  };
  auto copy8 = [](uint32_t dst, const float2 *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
  };
  // the pass's ops, descriptors and this set's matrices next to the tile: read
  // from global memory op by op they were a chain of three latencies each (and
  // they were uploaded before the call's first pass)
  pass_start();
  for (uint32_t k = threadIdx.x; k < (uint32_t)P.nops * kSitesEntry; k += T) {
    const uint32_t oi = k / kSitesEntry, w = k % kSitesEntry;
    const uint4 *op = reinterpret_cast<const uint4 *>(P.ops + oi);
    if (w < 2) {
      ent[k] = __ldg(op + w);
      continue;
    }
    const uint4 *d = reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(P.mats) + 16 * (size_t)P.ops[oi].mat);
    if (w < 8) {
      ent[k] = __ldg(d + (w - 2));
    } else {
      const int mat = reinterpret_cast<const int *>(d + 4)[(w - 8) / 2];
      if (mat >= 0) ent[k] = __ldg(reinterpret_cast<const uint4 *>(pm + mat) + (w & 1));
    }
  }
  pass_wait();
  for (uint32_t i = 0; i * T + threadIdx.x < nunits; i++) {
    const uint64_t g = goff(i);
    const uint32_t l = (i * T + threadIdx.x) * 2, a = swb<float>(l), b = swb<float>(l + 1);
    copy8(vs0 + a, &g0[g]);
    copy8(vs0 + b, &g0[g + 1]);
    if (TWO) {
      copy8(vs1 + a, &g1[g]);
      copy8(vs1 + b, &g1[g + 1]);
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  if (TWO && (P.flags & kPassShift)) {
    __syncthreads();
    shift_energy(reinterpret_cast<const float2 *>(smem_raw), reinterpret_cast<float2 *>(smem_raw) + TS, TS, acc + P.mat0);
  }
  if (!TWO && (P.flags & kPassNorm)) {
    const float p = warp_sum(loaded_norm(reinterpret_cast<const float2 *>(smem_raw), nunits));
    if ((threadIdx.x & 31) == 0) red[0][threadIdx.x >> 5] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0;
      for (uint32_t w = 0; w < (T + 31) / 32; w++) t += (double)red[0][w];
      atomicAdd(acc + P.mat0, t);
    }
  }
  for (int oi = 0; oi < P.nops; oi++) {
    __syncthreads();
    if (TWO && oi > 0) flush_probes(ent + (uint32_t)(oi - 1) * kSitesEntry, red[(oi - 1) & 1], acc);
    sites_op<TWO>(vs0, vs1, P.m, ent + (uint32_t)oi * kSitesEntry, red[oi & 1]);
  }
  __syncthreads();
  if (TWO) flush_probes(ent + (uint32_t)(P.nops - 1) * kSitesEntry, red[(P.nops - 1) & 1], acc);
  const float2 *v0 = reinterpret_cast<const float2 *>(smem_raw);
  for (uint32_t i = 0; i * T + threadIdx.x < nunits; i++) {
    const uint32_t l = (i * T + threadIdx.x) * 2;
    const uint64_t g = goff(i);
    __stcs(reinterpret_cast<int4 *>(&g0[g]), Unit<float>::get(v0, l));
    if (TWO) __stcs(reinterpret_cast<int4 *>(&g1[g]), Unit<float>::get(v0 + TS, l));
  }
}

// The pass is made of TOP_SITES ops only and they fit the staging area.
bool sites_pass_ok(const TilePass &p, const HostPass &h) {
  if (p.nops < 1 || p.nops > kMaxSitesOps) return false;
  for (int i = 0; i < p.nops; i++)
    if (h.ops[i].kind != TOP_SITES) return false;
  return true;
}

sv_status launch_tile_sites(sv_state *s, const TilePass &p, int batch, int threads, cudaStream_t stream) {
  const size_t smem = tile_smem(s->dt, p.m, (int)p.nvec) + (size_t)p.nops * kSitesEntry * 16;
  if (smem > (220u << 10)) return set_error(SV_EINVAL, "tile too large for shared memory");
  const dim3 grid((unsigned)(1ull << (p.n - p.m)), (unsigned)batch);
  const void *fn = p.nvec > 1 ? (const void *)k_tile_sites<true> : (const void *)k_tile_sites<false>;
  SV_TRY(func_attr_once(fn, s->device, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 << 10));
  SV_CUDA(launch_early(p.nvec > 1 ? k_tile_sites<true> : k_tile_sites<false>, grid, threads, smem, stream, p));
  g_launches++;
  return SV_OK;
}

}  // namespace sv
