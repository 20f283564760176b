// K8b: expectations of Pauli strings with X or Y factors, many x masks per
// pass over the state.
//
// Every string is Hermitian, so the terms of amplitudes x and x ^ xm are
// complex conjugates and a group (the strings sharing one x mask xm) needs
// each pair once:  2 sum_{pairs} Re(f(x) conj(psi[x ^ xm]) psi[x]),
// f(x) = sum_t c_t i^{k_t} (-1)^{popcount(x & z_t)}.
// A CTA loads a tile (the three lowest qubits and up to m - 3 chosen ones)
// into shared memory and evaluates every group whose x mask lies in the tile,
// so an n-qubit transverse field takes ceil((n - 3) / 10) reads of the state
// instead of one pass per qubit that reads the state twice.
//
// Strings of one X whose sign is the same over a tile (a transverse field)
// are taken KR at a time: a thread holds the 2^KR amplitudes of KR such
// qubits in registers, so one shared-memory read serves KR strings (one read
// per string was 2x the HBM time of a 13-qubit tile).  The others go pair by
// pair through shared memory.
//
// Bound: HBM and issue slots about equally (26 qubits, ten strings a pass:
// 128 us, 4.1 TB/s, 63% of issue slots; a pass of six 91 us).  13-qubit tiles
// (complex64, 64 KB) leave three CTAs per SM, whose loads and arithmetic
// overlap; larger tiles save no pass up to 33 qubits.  The 28-qubit
// transverse-field Ising energy: 31.4 ms (a pass per X string) -> 1.85 ms.
#include <algorithm>
#include <cstring>

#include "sv_device.cuh"
#include "sv_internal.h"

namespace sv {

constexpr int kXGroups = 64;      // groups per pass
constexpr int kXTerms = 128;      // their terms
constexpr int kXThreads = 256;
constexpr int kXRounds = 4;       // rounds per pass
constexpr int kXTrips = 16;       // 16-byte units per thread

template <typename R> struct XTileArgs {
  int32_t n, m, L, ng;
  int8_t hi_pos[16];              // qubit of tile bit L + j
  int8_t out_pos[kMaxQ];          // qubits outside the tile, ascending
  uint32_t xl[kXGroups];          // x mask in tile bits
  uint16_t t0[kXGroups + 1];      // terms of each group
  uint32_t zl[kXTerms];           // z mask in tile bits
  uint32_t odd[kXTerms];          // k_t odd: the term takes Im(conj(w) v)
  uint64_t gz[kXTerms];           // z mask outside the tile
  R c[kXTerms];                   // 2 c_t with the sign of i^{k_t}
  // rounds of KR single-X strings: tile bits held in registers, the positions
  // of the thread bits, and each string's coefficient and outside z mask
  int32_t nrounds;
  int8_t rbit[kXRounds][8];
  int8_t tpos[kXRounds][8];
  uint64_t rgz[kXRounds][8];
  R rc[kXRounds][8];
};
static_assert(sizeof(XTileArgs<double>) <= 8192, "kernel parameters");
template <typename R> constexpr int kXRegs = sizeof(R) == 4 ? 5 : 4;   // KR: 64 registers of amplitudes

// Sum of a tile's products in the state's precision, kept exactly enough to
// be added to the FP64 total once per tile: complex64 as an unevaluated pair
// of floats (two-sum, 48 bits), complex128 directly.
template <typename R> struct TileAcc;
template <> struct TileAcc<float> {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
    hi = s;
  }
  // (an infinite or NaN sum stays what it is: its error term is NaN)
  __device__ __forceinline__ double value() const { return isfinite(hi) ? (double)hi + (double)lo : (double)hi; }
};
template <> struct TileAcc<double> {
  double v = 0;
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ double value() const { return v; }
};

// Slot of tile amplitude l: complex64 keeps even/odd pairs together (16-byte
// copies) and XORs slot bits 1..3 with tile bits 4..6 and 8..10; complex128
// XORs bits 0..2 with bits 3..5 and 6..8.  Linear over GF(2).
template <typename R> __host__ __device__ __forceinline__ uint32_t xslot(uint32_t l) {
  return sizeof(R) == 4 ? l ^ ((((l >> 4) ^ (l >> 8)) & 7u) << 1) : l ^ (((l >> 3) ^ (l >> 6)) & 7u);
}

// acc + x * w, component by component
__device__ __forceinline__ void dot_acc(float2 x, float2 w, float2 &acc) {
  uint64_t r;
  asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n mov.b64 c, {%5, %6};\n"
      " fma.rn.f32x2 %0, a, b, c;\n}\n"
      : "=l"(r)
      : "f"(x.x), "f"(x.y), "f"(w.x), "f"(w.y), "f"(acc.x), "f"(acc.y));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(acc.x), "=f"(acc.y) : "l"(r));
}
__device__ __forceinline__ void dot_acc(double2 x, double2 w, double2 &acc) {
  acc.x = fma(x.x, w.x, acc.x);
  acc.y = fma(x.y, w.y, acc.y);
}

template <typename R>
__global__ void __launch_bounds__(kXThreads) k_expect_tile(const int4 *__restrict__ amps,
                                                           const __grid_constant__ XTileArgs<R> A, double *partial) {
  using C = typename Cx<R>::T;
  constexpr uint32_t APU = 16 / sizeof(C);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[kXThreads / 32];
  C *v = reinterpret_cast<C *>(smem_raw);
  const uint32_t TS = 1u << A.m, T = blockDim.x, nunits = TS / APU;
  const uint64_t ntiles = 1ull << (A.n - A.m);
  const uint32_t segmask = (1u << A.L) - 1;
  auto spread = [&](uint32_t l) -> uint64_t {
    uint64_t g = l & segmask;
    for (uint32_t x = l >> A.L; x; x &= x - 1) g |= 1ull << A.hi_pos[__ffs(x) - 1];
    return g;
  };
  const uint64_t gthr = spread(threadIdx.x * APU);
  // the trips' parts of a unit's state index and slot, shared by all threads
  // (computed per unit they were half of the kernel's instructions)
  __shared__ uint64_t s_trip[kXTrips];
  if (threadIdx.x < nunits / T) s_trip[threadIdx.x] = spread(threadIdx.x * T * APU);
  const uint32_t vs = smem_u32(v), sthr_u = xslot<R>(threadIdx.x * APU);
  __syncthreads();
  double acc = 0;
  for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    uint64_t base = 0;
    for (uint64_t t = tile; t; t &= t - 1) base |= 1ull << A.out_pos[__ffsll((long long)t) - 1];
    for (uint32_t i = 0; i < nunits / T; i++) {
      const uint64_t g = base | gthr | s_trip[i];
      const uint32_t slot = vs + (sthr_u ^ xslot<R>(i * T * APU)) * (uint32_t)sizeof(C);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(slot), "l"(amps + g / APU) : "memory");
    }
    cp_async_wait_all();
    __syncthreads();
    TileAcc<R> tot;
    constexpr int KR = kXRegs<R>, D = 1 << KR;
    for (int ri = 0; ri < A.nrounds; ri++) {
      uint32_t so[KR];
#pragma unroll
      for (int j = 0; j < KR; j++) so[j] = xslot<R>(1u << A.rbit[ri][j]);
      uint32_t l = 0;
#pragma unroll
      for (int i = 0; i < 8; i++) l |= ((threadIdx.x >> i) & 1u) << A.tpos[ri][i];
      if (threadIdx.x < (TS >> KR)) {
        const uint32_t s0 = xslot<R>(l);
        C x[D];
#pragma unroll
        for (int y = 0; y < D; y++) {
          uint32_t sl = s0;
#pragma unroll
          for (int j = 0; j < KR; j++) sl ^= ((y >> j) & 1) ? so[j] : 0u;
          x[y] = v[sl];
        }
#pragma unroll
        for (int j = 0; j < KR; j++) {
          const R c = A.rc[ri][j];
          if (c == R(0)) continue;
          C a = czero<C>();
#pragma unroll
          for (int y = 0; y < D; y++)
            if (!((y >> j) & 1)) dot_acc(x[y], x[y | (1 << j)], a);
          tot.add(((__popcll(base & A.rgz[ri][j]) & 1) ? -c : c) * (a.x + a.y));
        }
      }
    }
    for (int gi = 0; gi < A.ng; gi++) {
      const uint32_t xm = A.xl[gi];
      const int hb = 31 - __clz(xm);
      const uint32_t sx = xslot<R>(xm);
      const uint32_t lthr = ins0(threadIdx.x, hb), sthr = xslot<R>(lthr);
      const int t0 = A.t0[gi], t1 = A.t0[gi + 1];
      R part = 0;
      for (uint32_t p = 0; p < TS / 2; p += T) {
        const uint32_t lt = ins0(p, hb), l = lthr | lt;
        const uint32_t s0 = sthr ^ xslot<R>(lt);
        const C x = v[s0], w = v[s0 ^ sx];
        const R re = fma(w.x, x.x, w.y * x.y), im = fma(w.x, x.y, -(w.y * x.x));
        R fr = 0, fi = 0;
        for (int t = t0; t < t1; t++) {
          const bool neg = (__popc(l & A.zl[t]) + __popcll(base & A.gz[t])) & 1;
          const R c = neg ? -A.c[t] : A.c[t];
          if (A.odd[t]) fi += c;
          else fr += c;
        }
        part = fma(fr, re, fma(-fi, im, part));
      }
      tot.add(part);
    }
    acc += tot.value();
    __syncthreads();
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (uint32_t w = 0; w < (T + 31) / 32; w++) t += red[w];
    partial[blockIdx.x] = t;
  }
}

// Positions of a round's thread bits: the first four take tile bits that
// reach different banks (the vector each position adds to the 8- or 16-byte
// bank index under xslot, independent over GF(2)), so a wavefront's lanes do
// not collide; the rest follow in order.
template <typename R> static void thread_positions(uint32_t fixed, int m, int8_t *tpos) {
  const uint32_t banks = sizeof(R) == 4 ? 15u : 7u;
  uint32_t basis[4] = {0, 0, 0, 0}, used = fixed;
  int k = 0;
  for (int p = 0; p < m && k < 4; p++) {
    if ((used >> p) & 1u) continue;
    uint32_t x = xslot<R>(1u << p) & banks;
    for (int b = 3; b >= 0 && x; b--)
      if ((x >> b) & 1u) {
        if (!basis[b]) {
          basis[b] = x;
          used |= 1u << p;
          tpos[k++] = (int8_t)p;
          break;
        }
        x ^= basis[b];
      }
  }
  for (int p = 0; p < m && k < 8; p++)
    if (!((used >> p) & 1u)) tpos[k++] = (int8_t)p;
  for (; k < 8; k++) tpos[k] = 0;   // thread bits beyond the tile's groups are never set
}

// Tile size of the expectation passes: 13 qubits (complex128: 12, the same
// 64 KB), fewer for small states so that there is a tile for every SM.
static int xtile_m(const sv_state *s) { return std::min(s->dt == SV_C64 ? 13 : 12, std::max(8, s->n - 8)); }
constexpr int kXTileL = 3;

// A group of nt strings goes through tile passes when its x mask fits a tile
// next to the low qubits.  Below 10 qubits, and beyond 8 strings on one mask, the
// table kernel (k_expect) is used: its cost per amplitude does not grow with the
// strings.  From 22 qubits on (complex128 21), where amplitudes count more than launches, it is the
// better one beyond 4 strings, or 3 of the only group (26 qubits, complex64, eight
// groups of 3, 4 and 6: tiles 1.58, 1.91 and 2.71 ms, tables 2.04 to 2.06; one group
// of 3, 4 and 8: 268, 314 and 514 us, 300; 18 qubits, one of 8: 31 us and 43).
bool expect_tile_ok(const sv_state *s, uint64_t xm, int nt, bool only) {
  const int most = s->n <= (s->dt == SV_C64 ? 21 : 20) ? 8 : only ? 3 : 4;
  return s->n >= 10 && xm != 0 && nt <= most &&
         __builtin_popcountll(xm >> kXTileL) <= xtile_m(s) - kXTileL;
}

template <typename R>
static sv_status expect_tiles(sv_state *s, const sv_pauli_term *terms, const std::vector<std::vector<int>> &groups,
                              double *out_dev) {
  const int m = xtile_m(s), L = kXTileL, n = s->n;
  std::vector<size_t> order(groups.size());
  for (size_t i = 0; i < order.size(); i++) order[i] = i;
  auto xmask = [&](size_t g) { return terms[groups[g][0]].x_mask; };
  std::sort(order.begin(), order.end(), [&](size_t a, size_t b) { return xmask(a) < xmask(b); });
  std::vector<char> done(groups.size(), 0);
  size_t left = groups.size();
  const size_t smem = ((size_t)1 << m) * amp_bytes(s->dt);
  constexpr int KR = kXRegs<R>;
  // a unit per thread and trip (kXTrips at most: 2^m / APU / 2^(m - KR)), and
  // a group of 2^KR amplitudes per thread
  const int threads = std::max(64, std::min(kXThreads, 1 << (m - KR)));
  SV_TRY(func_attr_once((const void *)k_expect_tile<R>, s->device, cudaFuncAttributeMaxDynamicSharedMemorySize,
                        64 << 10));
  double *partial = reinterpret_cast<double *>(s->ws + kWsRed);
  const size_t cap = red_bytes(n) / sizeof(double);
  const int grid = (int)std::min<uint64_t>(1ull << (n - m), (uint64_t)s->sm_count * 3);
  size_t used = 0;
  while (left > 0) {
    XTileArgs<R> A;
    std::memset(&A, 0, sizeof(A));
    uint64_t S = (1ull << L) - 1;
    std::vector<size_t> mine;
    int nt = 0;
    for (size_t i : order) {
      if (done[i]) continue;
      const uint64_t x = xmask(i);
      if (__builtin_popcountll(S | x) > m || (int)mine.size() == kXGroups || nt + (int)groups[i].size() > kXTerms)
        continue;
      S |= x;
      nt += (int)groups[i].size();
      mine.push_back(i);
      done[i] = 1;
      left--;
    }
    for (int q = 0; q < n && __builtin_popcountll(S) < m; q++) S |= 1ull << q;
    int loc[64], k = 0, no = 0;
    for (int q = 0; q < n; q++) {
      if ((S >> q) & 1) {
        if (k >= L) A.hi_pos[k - L] = (int8_t)q;
        loc[q] = k++;
      } else {
        loc[q] = -1;
        A.out_pos[no++] = (int8_t)q;
      }
    }
    auto local = [&](uint64_t mask) {
      uint32_t l = 0;
      for (; mask; mask &= mask - 1) {
        const int q = __builtin_ctzll(mask);
        if (loc[q] >= 0) l |= 1u << loc[q];
      }
      return l;
    };
    A.n = n;
    A.m = m;
    A.L = L;
    // single X strings without z bits in the tile, KR to a round
    int t = 0, g = 0, ns = 0;
    std::vector<size_t> rest;
    for (size_t i : mine) {
      const sv_pauli_term &P = terms[groups[i][0]];
      if (groups[i].size() != 1 || __builtin_popcountll(P.x_mask) != 1 || (P.z_mask & S) || ns >= kXRounds * KR ||
          (R)(2.0 * P.coeff) == R(0)) {
        rest.push_back(i);
        continue;
      }
      A.rbit[ns / KR][ns % KR] = (int8_t)__builtin_ctz(local(P.x_mask));
      A.rgz[ns / KR][ns % KR] = P.z_mask & ~S;
      A.rc[ns / KR][ns % KR] = (R)(2.0 * P.coeff);
      ns++;
    }
    A.nrounds = (ns + KR - 1) / KR;
    for (int r = 0; r < A.nrounds; r++) {
      uint32_t bits = 0;
      const int have = std::min(KR, ns - r * KR);
      for (int j = 0; j < have; j++) bits |= 1u << A.rbit[r][j];
      for (int j = have, p = m - 1; j < KR; p--)   // fill the last round's registers with unused tile bits
        if (!((bits >> p) & 1u)) {
          bits |= 1u << p;
          A.rbit[r][j++] = (int8_t)p;
        }
      thread_positions<R>(bits, m, A.tpos[r]);
    }
    A.ng = (int)rest.size();
    for (; g < A.ng; g++) {
      const size_t gm = rest[g];
      A.xl[g] = local(xmask(gm));
      A.t0[g] = (uint16_t)t;
      for (int ti : groups[gm]) {
        const sv_pauli_term &P = terms[ti];
        const int ip = __builtin_popcountll(P.x_mask & P.z_mask) & 3;
        A.zl[t] = local(P.z_mask);
        A.gz[t] = P.z_mask & ~S;
        // Re(i^k c (re + i im)): c re, -c im, -c re, c im for k = 0..3; the
        // kernel subtracts the odd part
        A.odd[t] = (uint32_t)(ip & 1);
        A.c[t] = (R)((ip & 2) ? -2.0 * P.coeff : 2.0 * P.coeff);
        t++;
      }
    }
    A.t0[A.ng] = (uint16_t)t;
    if (used + (size_t)grid > cap) {   // the area is full: fold what it holds into its first value
      SV_TRY(launch_finalize(s, partial, (int)used, partial));
      used = 1;
    }
    k_expect_tile<R><<<grid, threads, smem, s->stream>>>(reinterpret_cast<const int4 *>(s->amps), A, partial + used);
    g_launches++;
    used += grid;
  }
  SV_CUDA(cudaGetLastError());
  return launch_finalize(s, partial, (int)used, out_dev);
}

sv_status launch_expect_tiles(sv_state *s, const sv_pauli_term *terms, const std::vector<std::vector<int>> &groups,
                              double *out_dev) {
  return s->dt == SV_C64 ? expect_tiles<float>(s, terms, groups, out_dev)
                         : expect_tiles<double>(s, terms, groups, out_dev);
}

}  // namespace sv
