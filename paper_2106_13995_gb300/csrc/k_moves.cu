// K15: runs of permutation gates (X, CNOT, Toffoli, SWAP, ...; paper Sec. III's
// reversible arithmetic) as one move of every amplitude.
//
// Table passes (K11) compose the gates of a 13-qubit tile; a 7-bit multiplier
// on 29 qubits takes 15 of them, a read and a write of the state each.  Here a
// run is cut where its gates move more than 22 qubits (21 for complex128): the
// state is a set of chunks of 2^22 amplitudes (32 MB, so that two of them stay
// in the L2 cache), and within a chunk every amplitude goes straight to its
// place.  One launch fills chunk j - 1 from one of two scratch buffers of the
// workspace and, in other CTAs, copies chunk j into the other buffer.
//
// Where an amplitude comes from is computed, not looked up: a thread follows 32
// of them through the run's gates (last one first) with a 32-bit word per index
// bit in shared memory, so a multi-controlled X is one AND and one XOR for all
// 32; a bit transpose then gives 32 indices.  Gates whose controls read 0 in
// qubits outside the chunk, or in qubits that no gate moves and that are fixed
// for the CTA, are left out CTA by CTA (half of a multiplier's).  The indices
// need no amplitudes: a launch starts computing them while the last one still
// moves its own (programmatic launch, and every CTA waits for the last launch
// before it reads or writes amplitudes or scratch).
//
// Bound: latency, of the words of the bit-sliced gates in shared memory and of a
// gather that reads 8 bytes from each of 32 lines a warp: no unit is full (load-
// store data pipe 50%, L2 41%, DRAM 26%, issue 30% with 37% of the warps; short
// scoreboard and MIO throttle are the top stalls).  A chunk of 32 MB takes 36 us, 10
// of them HBM.  The 7-bit multiplier on 29
// qubits took 15 table passes of 1.6 ms; its moves take 4.6 ms (6.4 with the
// launches one after the other, 5.9 with the copying CTAs first, 4.8 in chunks
// of 2^23).
#include <algorithm>
#include <cstring>
#include <vector>

#include "moves.cuh"
#include "sv_device.cuh"
#include "sv_internal.h"

namespace sv {

struct MoveArgs {
  uint64_t gbase, cbase;       // global offsets of the chunk to fill and of the one to copy
  const void *src;             // scratch that holds the chunk to fill
  void *dst;                   // scratch for the chunk to copy
  uint32_t fill, copy;         // tiles (CTAs) of each, equal or 0
};

__device__ __forceinline__ uint64_t move_spread(const TilePass &P, uint32_t loc) {
  uint64_t r = 0;
  for (; loc; loc &= loc - 1) r |= 1ull << P.hi_pos[__ffs(loc) - 1];
  return r;
}

template <typename C>
__global__ void __launch_bounds__(kMoveThreads, 7) k_moves(const __grid_constant__ TilePass P,
                                                           const __grid_constant__ MoveArgs A) {
  __shared__ uint32_t planes[kMovePlanes * kMoveThreads];
  __shared__ __align__(16) uint2 list[kMoveThreads + 8];   // padded to whole fours, and read four ahead
  __shared__ uint32_t counts[kMoveThreads / 32];
  __shared__ uint64_t off[32];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const bool copies = blockIdx.x >= A.fill;
  const uint32_t tile = copies ? blockIdx.x - A.fill : blockIdx.x;
  C *amps = reinterpret_cast<C *>(P.v0);
  pass_start();
  if (copies) {
    pass_wait();
    constexpr uint32_t APU = 16 / sizeof(C), kUnits = (1u << kMoveBits) / APU / kMoveThreads, kBatch = 8;
    if (tid < kUnits) off[tid] = move_spread(P, tid * kMoveThreads * APU);
    const uint64_t base = A.cbase | move_spread(P, (tile << kMoveBits) | (tid * APU));
    int4 *d = reinterpret_cast<int4 *>(static_cast<C *>(A.dst) + ((size_t)tile << kMoveBits)) + tid;
    __syncthreads();
#pragma unroll
    for (uint32_t i0 = 0; i0 < kUnits; i0 += kBatch) {
      int4 v[kBatch];
#pragma unroll
      for (uint32_t i = 0; i < kBatch; i++) v[i] = __ldcs(reinterpret_cast<const int4 *>(amps + (base | off[i0 + i])));
#pragma unroll
      for (uint32_t i = 0; i < kBatch; i++) d[(i0 + i) * kMoveThreads] = v[i];
    }
    return;
  }
  const unsigned char *blk = static_cast<const unsigned char *>(P.mats) + 16 * (size_t)P.mat0;
  const MoveDesc &D = *reinterpret_cast<const MoveDesc *>(blk);
  const MoveOp *ops = reinterpret_cast<const MoveOp *>(blk + sizeof(MoveDesc));
  const uint32_t cta = move_deposit(tile, D.ord, kMoveBits);
  const uint32_t loc = cta | lane | move_deposit(warp, D.ord, 10);
  const uint64_t known = A.gbase | move_spread(P, cta);
  if (tid < 32) off[tid] = move_spread(P, move_deposit(tid, D.ord, 5));
  // the planes of this thread's 32 places
  char *mine = reinterpret_cast<char *>(planes + tid);
  auto plane = [&](uint32_t o) -> uint32_t & { return *reinterpret_cast<uint32_t *>(mine + o); };
  const uint32_t pmask = D.pmask;
  for (uint32_t x = pmask; x; x &= x - 1) {
    const int i = __ffs(x) - 1;
    plane(D.plane[i]) = (loc >> i) & 1u ? ~0u : 0u;
  }
#pragma unroll
  for (int k = 0; k < 5; k++)
    if ((pmask >> D.ord[5 + k]) & 1u) plane(D.plane[D.ord[5 + k]]) = word_pattern(k);
  plane(D.ones) = ~0u;
  auto step = [&](uint32_t x, uint32_t y) {
    const uint32_t f = plane(x >> 16) & plane(y & 0xffffu);
    uint32_t &t = plane(x & 0xffffu);
    t = (t & (uint32_t)((int32_t)y >> 16)) ^ f;
  };
  const uint32_t nops = D.nops;
  for (uint32_t b = 0; b < nops; b += kMoveThreads) {
    // the batch's gates that act in this CTA, in order
    const bool in = b + tid < nops;
    int4 o = make_int4(0, 0, 0, 0);
    if (in) o = __ldg(reinterpret_cast<const int4 *>(ops + b + tid));
    const uint64_t gate = (uint64_t)(uint32_t)o.x | ((uint64_t)(uint32_t)o.y << 32);
    const bool act = in && (known & gate) == gate;
    const uint32_t votes = __ballot_sync(~0u, act);
    __syncthreads();   // the last batch's list has been read
    if (lane == 0) counts[warp] = __popc(votes);
    __syncthreads();
    uint32_t at = __popc(votes & ((1u << lane) - 1u)), n = 0;
#pragma unroll
    for (uint32_t w = 0; w < kMoveThreads / 32; w++) {
      at += w < warp ? counts[w] : 0u;
      n += counts[w];
    }
    if (act) list[at] = make_uint2((uint32_t)o.z, (uint32_t)o.w);
    if (tid < 4) list[n + tid] = make_uint2(D.idle | ((uint32_t)D.idle << 16), D.idle | 0xffff0000u);
    __syncthreads();
    const uint4 *l4 = reinterpret_cast<const uint4 *>(list);
    uint4 e0 = l4[0], e1 = l4[1];
    for (uint32_t k = 0; k < n; k += 4) {
      const uint4 d0 = e0, d1 = e1;
      e0 = l4[k / 2 + 2];
      e1 = l4[k / 2 + 3];
      step(d0.x, d0.y);
      step(d0.z, d0.w);
      step(d1.x, d1.y);
      step(d1.z, d1.w);
    }
  }
  uint32_t r[32];
#pragma unroll
  for (int i = 0; i < 32; i++) r[i] = (pmask >> i) & 1u ? plane(D.plane[i]) : 0u;
  transpose32(r);
  const uint32_t rest = loc & ~pmask;
  const C *src = static_cast<const C *>(A.src);
  C *dst = amps + (A.gbase | move_spread(P, loc));
  pass_wait();   // (the indices needed no memory of the last launch)
  constexpr int kBatch = 128 / sizeof(C);   // 32 registers of loads in flight
#pragma unroll
  for (int i0 = 0; i0 < 32; i0 += kBatch) {
    C v[kBatch];
#pragma unroll
    for (int i = 0; i < kBatch; i++) v[i] = __ldcg(src + (r[i0 + i] | rest));
#pragma unroll
    for (int i = 0; i < kBatch; i++) __stcs(dst + off[i0 + i], v[i]);
  }
}

sv_status launch_moves(sv_state *s, const TilePass &p, cudaStream_t stream) {
  const size_t chunk = ((size_t)1 << p.m) * amp_bytes(s->dt);
  const uint64_t chunks = 1ull << (p.n - p.m);
  if (p.m < kMoveBits || p.m > moves_m(s->n, s->dt) || s->ws_bytes < moves_off(s->n) + moves_bytes(s->n, s->dt))
    return set_error(SV_EINVAL, "internal: permutation run without its scratch");
  char *scratch = s->ws + moves_off(s->n);
  auto base_of = [&](uint64_t j) {
    uint64_t r = 0;
    for (int k = 0; j >> k; k++) r |= ((j >> k) & 1ull) << p.out_pos[k];
    return r;
  };
  const uint32_t tiles = 1u << (p.m - kMoveBits);
  for (uint64_t j = 0; j <= chunks; j++) {
    MoveArgs A;
    A.copy = j < chunks ? tiles : 0;
    A.fill = j > 0 ? tiles : 0;
    A.cbase = j < chunks ? base_of(j) : 0;
    A.gbase = j > 0 ? base_of(j - 1) : 0;
    A.dst = scratch + (j & 1) * chunk;
    A.src = scratch + ((j + 1) & 1) * chunk;
    SV_CUDA(launch_early(s->dt == SV_C64 ? k_moves<float2> : k_moves<double2>, dim3(A.copy + A.fill), kMoveThreads, 0,
                         stream, p, A));
    g_launches++;
  }
  return SV_OK;
}

// ---------------------------------------------------------------------------
// host: gates to multi-controlled X, runs to passes
// ---------------------------------------------------------------------------
// A permutation of 2^k values as multi-controlled X, appended in order (the
// transformation-based synthesis of Miller, Maslov and Dueck, DAC 2003: values
// are put right in increasing order by gates that leave smaller ones alone).
void perm_to_moves(const int *perm, int k, const std::vector<int> &q, uint64_t controls, std::vector<Move> &out) {
  std::vector<int> p(perm, perm + (1 << k));
  std::vector<std::pair<int, int>> gates;   // (control mask, target bit), applied to the outputs
  auto apply = [&](int cm, int t) {
    for (int &v : p)
      if ((v & cm) == cm) v ^= 1 << t;
    gates.push_back({cm, t});
  };
  for (int i = 0; i < (1 << k); i++) {
    for (int b = 0; b < k; b++)
      if (((i & ~p[i]) >> b) & 1) apply(p[i], b);
    for (int b = 0; b < k; b++)
      if (((p[i] & ~i) >> b) & 1) apply(p[i] & ~(1 << b), b);
  }
  for (size_t g = gates.size(); g-- > 0;) {
    Move m{controls, q[gates[g].second]};
    for (int b = 0; b < k; b++)
      if ((gates[g].first >> b) & 1) m.controls |= 1ull << q[b];
    out.push_back(m);
  }
}

bool gate_moves(const Gate &g, std::vector<Move> &out) {
  const int k = (int)g.targets.size();
  int perm[8];
  if (k < 1 || k > 3 || g.inst >= 0 || g.param >= 0 || g.grad_gen > 0 || g.fixed_structure ||
      !permutation_of(g.U, k, perm))
    return false;
  uint64_t c = 0;
  for (int q : g.controls) c |= 1ull << q;
  perm_to_moves(perm, k, g.targets, c, out);
  return true;
}

// Moves of a run, in passes that move at most m - 5 qubits beyond the lowest
// five.  A move joins a pass when it commutes with the moves left for later
// ones: neither's target is the other's control.
std::vector<std::vector<Move>> plan_moves(const std::vector<Move> &moves, int m) {
  std::vector<std::vector<Move>> passes;
  std::vector<Move> left = moves;
  while (!left.empty()) {
    std::vector<Move> now, later;
    uint64_t in = 31, later_t = 0, later_c = 0;
    for (const Move &mv : left) {
      const uint64_t t = 1ull << mv.target;
      if (!(mv.controls & later_t) && !(t & later_c) && __builtin_popcountll(in | t) <= m) {
        in |= t;
        now.push_back(mv);
      } else {
        later_t |= t;
        later_c |= mv.controls;
        later.push_back(mv);
      }
    }
    passes.push_back(std::move(now));
    left.swap(later);
  }
  return passes;
}

// A pass of moves on n qubits with chunks of 2^m amplitudes: descriptor and ops
// into the matrix pool.
void emit_moves(DeviceProgram &prog, const std::vector<Move> &moves, int n, int m, std::vector<uint32_t> &op0s) {
  uint64_t moved = 0, in = 31;
  for (const Move &mv : moves) moved |= 1ull << mv.target;
  in |= moved;
  for (int q = 0; q < n && __builtin_popcountll(in) < m; q++) in |= 1ull << q;
  TilePass tp;
  std::memset(&tp, 0, sizeof(tp));
  tp.n = n;
  tp.m = m;
  tp.nvec = 1;
  tp.flags = kPassMoves;
  int local[64], ni = 0, no = 0;
  for (int q = 0; q < n; q++)
    if ((in >> q) & 1) {
      local[q] = ni;
      tp.hi_pos[ni++] = (int8_t)q;
    } else {
      tp.out_pos[no++] = (int8_t)q;
    }
  MoveDesc D;
  std::memset(&D, 0, sizeof(D));
  // lane bits: the lowest qubits (256-byte stores); word and warp bits: moved
  // qubits first, so that as many unmoved ones as possible are fixed for a CTA
  int no2 = 0;
  for (int i = 0; i < 5; i++) D.ord[no2++] = (uint8_t)i;
  for (int pass = 0; pass < 2; pass++)
    for (int i = 5; i < m; i++)
      if (((moved >> tp.hi_pos[i]) & 1) == (pass == 0 ? 1u : 0u)) D.ord[no2++] = (uint8_t)i;
  uint64_t known = ~in;
  for (int k = kMoveBits; k < m; k++) {
    const uint64_t q = 1ull << tp.hi_pos[D.ord[k]];
    if (!(moved & q)) known |= q;
  }
  int np = 0;
  for (int i = 0; i < 32; i++) {
    D.plane[i] = 0xffff;
    if (i >= m || ((known >> tp.hi_pos[i]) & 1)) continue;
    D.plane[i] = (uint16_t)(np++ * kMovePlaneBytes);
    D.pmask |= 1u << i;
  }
  D.ones = (uint16_t)(np * kMovePlaneBytes);
  D.tmp = (uint16_t)((np + 1) * kMovePlaneBytes);
  D.idle = (uint16_t)((np + 2) * kMovePlaneBytes);
  std::vector<MoveOp> ops;
  for (size_t k = moves.size(); k-- > 0;) {
    const Move &mv = moves[k];
    std::vector<uint16_t> c;
    for (uint64_t x = mv.controls & ~known; x; x &= x - 1) c.push_back(D.plane[local[__builtin_ctzll(x)]]);
    while (c.size() < 2) c.push_back(D.ones);
    const uint64_t gate = mv.controls & known;
    while (c.size() > 2) {   // two controls into one
      ops.push_back({gate, D.tmp, c[c.size() - 1], c[c.size() - 2], 0});
      c.pop_back();
      c.back() = D.tmp;
    }
    ops.push_back({gate, D.plane[local[mv.target]], c[0], c[1], 0xffff});
  }
  D.nops = (uint32_t)ops.size();
  while (prog.mats.size() % 16) prog.mats.push_back(0);
  tp.mat0 = (uint32_t)(prog.mats.size() / 16);
  const uint8_t *d = reinterpret_cast<const uint8_t *>(&D), *q = reinterpret_cast<const uint8_t *>(ops.data());
  prog.mats.insert(prog.mats.end(), d, d + sizeof(D));
  prog.mats.insert(prog.mats.end(), q, q + ops.size() * sizeof(MoveOp));
  op0s.push_back((uint32_t)prog.ops.size());
  prog.passes.push_back(tp);
}

// ---------------------------------------------------------------------------
// product states
// ---------------------------------------------------------------------------
// K16: amplitude x = product over q of v[q][bit q of x], written once.  Factors
// of six bits at a time come from tables (FP64, built once per persistent CTA);
// a chunk of 2^12 amplitudes multiplies its upper factors into one table in
// FP64, and an amplitude is one product of two entries in the state's type (one
// FP64 product each would be bound by the FP64 pipe).  The Hadamards in front of
// the 29-qubit multiplier took a tile pass of 3.4 ms (FP32-bound, 128
// multiply-adds an amplitude), the product 0.7 ms.
constexpr int kProdTables = 6;   // of six bits: 36 >= 34 qubits
struct ProductArgs {
  double2 v[6 * kProdTables][2];
};
template <typename R>
__global__ void __launch_bounds__(256) k_product(typename Cx<R>::T *__restrict__ a, uint64_t nchunks,
                                                 const __grid_constant__ ProductArgs A) {
  using C = typename Cx<R>::T;
  __shared__ double2 tab[kProdTables][64];
  __shared__ __align__(16) C low[64], up[2][64];
  const uint32_t tid = threadIdx.x;
  for (uint32_t e = tid; e < kProdTables * 64; e += 256) {
    double2 p = make_double2(1.0, 0.0);
    for (uint32_t b = 0; b < 6; b++) p = cmul(A.v[6 * (e >> 6) + b][(e >> b) & 1u], p);
    tab[e >> 6][e & 63u] = p;
  }
  __syncthreads();
  auto cast = [](double2 p) {
    C c;
    c.x = (R)p.x;
    c.y = (R)p.y;
    return c;
  };
  if (tid < 64) low[tid] = cast(tab[0][tid]);
  int turn = 0;
  for (uint64_t c = blockIdx.x; c < nchunks; c += gridDim.x, turn ^= 1) {
    if (tid < 64) {
      double2 p = tab[1][tid];
      for (int k = 2; k < kProdTables; k++) p = cmul(tab[k][(c >> (6 * (k - 2))) & 63u], p);
      up[turn][tid] = cast(p);
    }
    __syncthreads();   // (the table of the chunk before last has been read)
    constexpr uint32_t APU = 16 / sizeof(C), kTrips = 4096 / APU / 256;
#pragma unroll
    for (uint32_t i = 0; i < kTrips; i++) {
      const uint32_t x = (tid + 256 * i) * APU;
      __align__(16) C o[APU];
#pragma unroll
      for (uint32_t j = 0; j < APU; j++) o[j] = cmul(up[turn][x >> 6], low[(x & 63u) + j]);
      __stcs(reinterpret_cast<int4 *>(a + (c << 12) + x), *reinterpret_cast<const int4 *>(o));
    }
  }
}

bool product_of(const std::vector<Gate> &gates, int n, std::vector<cd> &U) {
  U.assign(4 * (size_t)n, cd(0.0));
  for (int q = 0; q < n; q++) U[4 * q] = U[4 * q + 3] = 1.0;
  for (const Gate &g : gates) {
    if (g.targets.size() != 1 || !g.controls.empty() || g.inst >= 0 || g.param >= 0 || g.grad_gen > 0 ||
        g.fixed_structure)
      return false;
    cd *u = &U[4 * (size_t)g.targets[0]];
    const cd a = u[0], b = u[1], c = u[2], d = u[3];
    u[0] = g.U[0] * a + g.U[1] * c;
    u[1] = g.U[0] * b + g.U[1] * d;
    u[2] = g.U[2] * a + g.U[3] * c;
    u[3] = g.U[2] * b + g.U[3] * d;
  }
  return true;
}

sv_status launch_product(sv_state *s, const TilePass &p, const HostPass &host, cudaStream_t stream) {
  if (!s->basis_known || s->n < 12) return set_error(SV_EINVAL, "internal: product pass on an unknown state");
  ProductArgs A;
  const double *u = reinterpret_cast<const double *>(host.mats + 16 * (size_t)p.mat0);
  for (int q = 0; q < 6 * kProdTables; q++)
    for (int r = 0; r < 2; r++) {
      if (q < s->n) {
        const double *e = u + 8 * q + 4 * r + 2 * ((s->basis_index >> q) & 1);   // row r, column: the basis bit
        A.v[q][r] = make_double2(e[0], e[1]);
      } else {
        A.v[q][r] = make_double2(1.0, 0.0);
      }
    }
  // the basis state's own phase, into a qubit's two factors
  for (int r = 0; r < 2; r++) {
    const cd v = cd(A.v[0][r].x, A.v[0][r].y) * s->basis_amp;
    A.v[0][r] = make_double2(v.real(), v.imag());
  }
  const uint64_t chunks = 1ull << (s->n - 12);
  const unsigned grid = (unsigned)std::min<uint64_t>(chunks, (uint64_t)s->sm_count * 8);
  if (s->dt == SV_C64)
    k_product<float><<<grid, 256, 0, stream>>>(reinterpret_cast<float2 *>(p.v0), chunks, A);
  else
    k_product<double><<<grid, 256, 0, stream>>>(reinterpret_cast<double2 *>(p.v0), chunks, A);
  g_launches++;
  SV_CUDA(cudaGetLastError());
  return SV_OK;
}

}  // namespace sv
