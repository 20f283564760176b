// Host run of permutation runs (test only): the moves of a gate list, cut into
// passes and emitted as the library does, then followed index by index as the
// kernel does.  src[x]: where the amplitude at x comes from, over all passes.
#include <cstring>
#include <vector>

#include "../../paper_2106_13995_gb300/csrc/moves.cuh"
#include "../../paper_2106_13995_gb300/csrc/sv_internal.h"

using namespace sv;

// Gate g: k[g] targets and nc[g] controls in q (targets first), perm 8 values.
// Returns the number of passes, or a negative error.
extern "C" int moves_emulate(int n, int m, int ngates, const int *k, const int *nc, const int *q, const int *perm,
                             uint32_t *src) {
  std::vector<Move> moves;
  for (int g = 0; g < ngates; g++) {
    Gate G;
    G.targets.assign(q, q + k[g]);
    G.controls.assign(q + k[g], q + k[g] + nc[g]);
    q += k[g] + nc[g];
    const int d = 1 << k[g];
    G.U.assign((size_t)d * d, cd(0.0));
    for (int c = 0; c < d; c++) G.U[(size_t)perm[8 * g + c] * d + c] = 1.0;
    if (!gate_moves(G, moves)) return -1;
  }
  const std::vector<std::vector<Move>> passes = plan_moves(moves, m);
  DeviceProgram prog;
  std::vector<uint32_t> op0s;
  for (const auto &p : passes) emit_moves(prog, p, n, m, op0s);
  const size_t N = (size_t)1 << n;
  std::vector<uint32_t> now(N), next(N);
  for (size_t i = 0; i < N; i++) now[i] = (uint32_t)i;
  for (const TilePass &P : prog.passes) {
    const uint8_t *blk = prog.mats.data() + 16 * (size_t)P.mat0;
    MoveDesc D;
    std::memcpy(&D, blk, sizeof(D));
    const MoveOp *ops = reinterpret_cast<const MoveOp *>(blk + sizeof(D));
    if (D.idle + kMovePlaneBytes > kMovePlanes * kMovePlaneBytes || P.m != m || m < kMoveBits) return -2;
    for (int k = 0; k < 5; k++)
      if (P.hi_pos[k] != k || D.ord[k] != k) return -3;
    auto spread = [&](uint32_t l) {
      uint32_t r = 0;
      for (int i = 0; i < m; i++) r |= ((l >> i) & 1u) << P.hi_pos[i];
      return r;
    };
    std::vector<char> hit(N, 0);
    for (uint32_t chunk = 0; chunk < 1u << (n - m); chunk++) {
      uint32_t gbase = 0;
      for (int k = 0; k < n - m; k++) gbase |= ((chunk >> k) & 1u) << P.out_pos[k];
      for (uint32_t tile = 0; tile < 1u << (m - kMoveBits); tile++) {
        const uint32_t cta = move_deposit(tile, D.ord, kMoveBits);
        const uint64_t known = gbase | spread(cta);
        for (uint32_t tid = 0; tid < (uint32_t)kMoveThreads; tid++) {
          const uint32_t loc = cta | (tid & 31u) | move_deposit(tid >> 5, D.ord, 10);
          uint32_t plane[kMovePlanes] = {0};
          auto at = [&](uint32_t o) -> uint32_t & { return plane[o / kMovePlaneBytes]; };
          for (int i = 0; i < m; i++)
            if ((D.pmask >> i) & 1u) at(D.plane[i]) = (loc >> i) & 1u ? ~0u : 0u;
          for (int k = 0; k < 5; k++)
            if ((D.pmask >> D.ord[5 + k]) & 1u) at(D.plane[D.ord[5 + k]]) = word_pattern(k);
          at(D.ones) = ~0u;
          for (uint32_t o = 0; o < D.nops; o++) {
            if ((known & ops[o].gate) != ops[o].gate) continue;
            const uint32_t f = at(ops[o].c1) & at(ops[o].c2);
            at(ops[o].t) = (ops[o].keep ? at(ops[o].t) : 0u) ^ f;
          }
          uint32_t r[32];
          for (int i = 0; i < 32; i++) r[i] = (D.pmask >> i) & 1u ? at(D.plane[i]) : 0u;
          transpose32(r);
          for (uint32_t w = 0; w < 32; w++) {
            const uint32_t to = gbase | spread(loc | move_deposit(w, D.ord, 5)), l = r[w] | (loc & ~D.pmask);
            if (l >> m || hit[to]++) return -4;
            next[to] = now[gbase | spread(l)];
          }
        }
      }
    }
    now.swap(next);
  }
  std::memcpy(src, now.data(), N * sizeof(uint32_t));
  return (int)prog.passes.size();
}
