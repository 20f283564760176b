// Gate fusion and tile-pass planning (host, FP64).
//
// Fusion: consecutive gates acting on at most K qubits are multiplied into one
// 2^K x 2^K block.  A gate joins the latest block that touches any of its
// qubits, so it only ever moves past blocks on disjoint qubits (which commute
// with it).  Products are formed in FP64 and cast to the state's type later.
//
// Pass planning: each pass holds a set S of tile qubits (the L lowest qubits
// plus chosen high ones, |S| = m).  Blocks whose targets lie in S are applied
// to 2^m-amplitude tiles in shared memory, so the pass reads and writes the
// state once.  A block that cannot join blocks every qubit it touches for the
// rest of the scan, which keeps every reordering between commuting blocks.
#include <algorithm>

#include "sv_internal.h"

namespace sv {

static int index_of(const std::vector<int> &v, int q) {
  for (size_t i = 0; i < v.size(); i++)
    if (v[i] == q) return (int)i;
  return -1;
}

// Embed a (controlled) gate on `targets`/`controls` into a dense matrix over
// the qubit list `Q` (which contains all of them).
template <typename T>
static std::vector<T> embed(const std::vector<T> &U, const std::vector<int> &targets,
                            const std::vector<int> &controls, const std::vector<int> &Q) {
  const int kq = (int)Q.size();
  const int D = 1 << kq;
  const int d = 1 << (int)targets.size();
  std::vector<int> tpos(targets.size()), cpos(controls.size());
  for (size_t j = 0; j < targets.size(); j++) tpos[j] = index_of(Q, targets[j]);
  for (size_t j = 0; j < controls.size(); j++) cpos[j] = index_of(Q, controls[j]);
  int tmask = 0, cmask = 0;
  for (int p : tpos) tmask |= 1 << p;
  for (int p : cpos) cmask |= 1 << p;
  std::vector<T> E((size_t)D * D, T(0.0));
  for (int col = 0; col < D; col++) {
    if ((col & cmask) != cmask) {
      E[(size_t)col * D + col] = T(1.0);
      continue;
    }
    int ct = 0;
    for (size_t j = 0; j < tpos.size(); j++) ct |= ((col >> tpos[j]) & 1) << j;
    for (int rt = 0; rt < d; rt++) {
      int row = col & ~tmask;
      for (size_t j = 0; j < tpos.size(); j++) row |= ((rt >> j) & 1) << tpos[j];
      E[(size_t)row * D + col] = U[(size_t)rt * d + ct];
    }
  }
  return E;
}

template <typename T>
static std::vector<T> matmul(const std::vector<T> &A, const std::vector<T> &B, int D) {
  std::vector<T> C((size_t)D * D, T(0.0));
  for (int i = 0; i < D; i++)
    for (int k = 0; k < D; k++) {
      const T a = A[(size_t)i * D + k];
      if (a == T(0.0)) continue;
      for (int j = 0; j < D; j++) C[(size_t)i * D + j] += a * B[(size_t)k * D + j];
    }
  return C;
}

static bool is_diagonal(const std::vector<cd> &U, int k) {
  const int d = 1 << k;
  for (int r = 0; r < d; r++)
    for (int c = 0; c < d; c++)
      if (r != c && U[(size_t)r * d + c] != cd(0.0)) return false;
  return true;
}

static std::vector<double> magnitudes(const std::vector<cd> &U) {
  std::vector<double> m(U.size());
  for (size_t e = 0; e < U.size(); e++) m[e] = std::abs(U[e]);
  return m;
}

// M over the qubits Q, multiplied from the left by a gate's entry magnitudes.
static void gate_magnitudes(const Gate &g, const std::vector<int> &Q, std::vector<double> &M) {
  const int D = 1 << (int)Q.size(), d = 1 << (int)g.targets.size();
  int cmask = 0, off[64], tmask = 0;
  for (int q : g.controls) cmask |= 1 << index_of(Q, q);
  for (int y = 0; y < d; y++) {
    off[y] = 0;
    for (size_t j = 0; j < g.targets.size(); j++) off[y] |= ((y >> j) & 1) << index_of(Q, g.targets[j]);
    tmask |= off[y];
  }
  double m[64 * 64], rows[64 * 64];
  for (int e = 0; e < d * d; e++) m[e] = std::abs(g.U[e]);
  for (int base = 0; base < D; base++) {
    if ((base & tmask) || (base & cmask) != cmask) continue;
    for (int y = 0; y < d; y++) std::copy_n(&M[(size_t)(base | off[y]) * D], D, rows + (size_t)y * D);
    for (int r = 0; r < d; r++) {
      double *to = &M[(size_t)(base | off[r]) * D];
      std::fill(to, to + D, 0.0);
      for (int y = 0; y < d; y++) {
        const double a = m[r * d + y];
        if (a == 0) continue;
        for (int c = 0; c < D; c++) to[c] += a * rows[(size_t)y * D + c];
      }
    }
  }
}

std::vector<Block> fuse(const std::vector<Gate> &gates, int K, bool mags) {
  std::vector<Block> blocks;
  blocks.reserve(gates.size());
  std::vector<int> last(64, -1);
  for (const Gate &g : gates) {
    std::vector<int> Q = g.targets;
    Q.insert(Q.end(), g.controls.begin(), g.controls.end());
    const bool standalone = K <= 1 || g.fixed_structure || g.grad_gen > 0 ||
                            g.controls.size() >= 2 || (int)Q.size() > K;
    int bstar = -1;
    for (int q : Q) bstar = std::max(bstar, last[q]);
    if (!standalone && bstar >= 0 && blocks[bstar].fusable) {
      Block &b = blocks[bstar];
      std::vector<int> uni = b.qubits;
      for (int q : Q)
        if (index_of(uni, q) < 0) uni.push_back(q);
      if ((int)uni.size() <= K) {
        const int D = 1 << (int)uni.size();
        const std::vector<cd> Ug = embed(g.U, g.targets, g.controls, uni);
        if (uni.size() > b.qubits.size()) b.U = embed(b.U, b.qubits, {}, uni);
        b.U = matmul(Ug, b.U, D);
        if (mags) {
          if (uni.size() > b.qubits.size()) b.mag = embed(b.mag, b.qubits, {}, uni);
          gate_magnitudes(g, uni, b.mag);
        }
        b.qubits = uni;
        // the block's older qubits may already have later blocks: keep those
        for (int q : uni) last[q] = std::max(last[q], bstar);
        continue;
      }
    }
    Block nb;
    if (g.grad_gen > 0) {
      nb.kind = TOP_GRAD;
      nb.qubits = g.targets;
      nb.gen = g.grad_gen;
      nb.slot = g.grad_slot;
      nb.fusable = false;
      nb.vmask = 3;
    } else if (standalone) {
      nb.qubits = g.targets;
      nb.controls = g.controls;
      nb.U = g.U;
      // a block that keeps explicit controls cannot absorb more gates
      nb.fusable = !g.fixed_structure && g.controls.empty() && K > 1;
      nb.param = g.fixed_structure ? g.param : -1;
      nb.param_gate = g.fixed_structure ? g.param_gate : -1;
      nb.inst = g.fixed_structure ? g.inst : -1;
      if (K <= 1) nb.fusable = false;
    } else {
      nb.qubits = Q;
      nb.U = embed(g.U, g.targets, g.controls, Q);
    }
    if (mags) nb.mag = magnitudes(nb.U);
    blocks.push_back(std::move(nb));
    const int idx = (int)blocks.size() - 1;
    for (int q : Q) last[q] = idx;
  }
  for (Block &b : blocks)
    if (b.kind == TOP_DENSE) b.diag = b.inst < 0 && is_diagonal(b.U, (int)b.qubits.size());
  return blocks;
}

static uint64_t qmask(const std::vector<int> &v) {
  uint64_t m = 0;
  for (int q : v) m |= 1ull << q;
  return m;
}

static int mat_entries(const Block &b) {
  if (b.kind == TOP_TC) return 1024;   // a 5-qubit block (its packed operand is counted as 32 x 32)
  if (b.kind != TOP_DENSE && b.kind != TOP_DIAG) return 0;
  const int d = 1 << (int)b.qubits.size();
  return b.diag ? d : d * d;
}

int max_targets(const std::vector<Block> &blocks) {
  int k = 0;
  for (const Block &b : blocks) k = std::max(k, (int)b.qubits.size());
  return k;
}

bool fit_tile(const std::vector<Block> &blocks, int n, int lmin, int mmax, int &m, int &L) {
  const int kmax = max_targets(blocks);
  m = std::min(m, n);
  if (m >= n) {
    L = std::min(L, n);
    return true;
  }
  if (m - kmax < lmin) m = std::min(n, std::min(mmax, kmax + lmin));
  if (m >= n) {
    m = n;
    L = std::min(L, n);
    return true;
  }
  L = std::min(L, m - kmax);
  return L >= lmin;
}

std::vector<PassPlan> plan_passes(std::vector<Block> blocks, int n, int m, int L,
                                  int max_ops, int max_mat_entries) {
  std::vector<PassPlan> passes;
  m = std::min(m, n);
  L = std::min(L, m);
  // every block must fit next to the L fixed low qubits
  if (m < n && max_targets(blocks) > m - L) return passes;
  const uint64_t low = (L >= 64) ? ~0ull : ((1ull << L) - 1);
  const uint64_t all = (n >= 64) ? ~0ull : ((1ull << n) - 1);
  std::vector<char> done(blocks.size(), 0);
  size_t remaining = blocks.size(), first = 0;
  while (remaining > 0) {
    while (first < blocks.size() && done[first]) first++;
    uint64_t S = low, blocked = 0;
    int nops = 0, nmat = 0;
    PassPlan P;
    for (size_t i = first; i < blocks.size(); i++) {
      if (done[i]) continue;
      Block &b = blocks[i];
      const uint64_t need = qmask(b.qubits);
      const uint64_t touch = need | qmask(b.controls) | b.xmask;
      if (touch & blocked) {
        blocked |= touch;
      } else if (__builtin_popcountll(S | need) <= m && nops < max_ops &&
                 nmat + mat_entries(b) <= max_mat_entries) {
        S |= need;
        nops++;
        nmat += mat_entries(b);
        P.ops.push_back(std::move(b));
        done[i] = 1;
        remaining--;
      } else {
        blocked |= touch;
      }
      if ((blocked & all) == all) break;
    }
    if (P.ops.empty()) return {};     // nothing fits: the caller reports it
    // fill the tile up to m qubits with the lowest unused qubits
    for (int q = 0; q < n && __builtin_popcountll(S) < m; q++) S |= 1ull << q;
    for (int q = 0; q < n; q++)
      if ((S >> q) & 1) P.S.push_back(q);
    passes.push_back(std::move(P));
  }
  return passes;
}

// Merge small blocks inside each pass: a block joins an earlier block of the
// same pass when every block between them acts on other qubits (so it may
// move back next to it) and the two together touch at most K qubits.  The
// product is formed in FP64 as in fuse().  Blocks with controls, parameters
// or non-dense kinds neither merge nor move past blocks sharing a qubit.
static bool mergeable(const Block &b) {
  return b.kind == TOP_DENSE && b.controls.empty() && b.param < 0 && b.inst < 0 && b.fusable;
}
std::vector<Block> merge_in_passes(std::vector<PassPlan> passes, int K) {
  std::vector<Block> out;
  for (PassPlan &P : passes) {
    std::vector<Block> &ops = P.ops;
    std::vector<char> alive(ops.size(), 1);
    for (size_t j = 0; j < ops.size(); j++) {
      if (!mergeable(ops[j])) continue;
      const uint64_t tj = qmask(ops[j].qubits);
      for (size_t i = j; i-- > 0;) {
        if (!alive[i]) continue;
        const uint64_t ti = qmask(ops[i].qubits) | qmask(ops[i].controls) | ops[i].xmask;
        if (mergeable(ops[i]) && __builtin_popcountll(qmask(ops[i].qubits) | tj) <= K) {
          Block &A = ops[i];
          std::vector<int> uni = A.qubits;
          for (int q : ops[j].qubits)
            if (index_of(uni, q) < 0) uni.push_back(q);
          const int D = 1 << (int)uni.size();
          const std::vector<cd> Ua = embed(A.U, A.qubits, {}, uni);
          const std::vector<cd> Ub = embed(ops[j].U, ops[j].qubits, {}, uni);
          A.U = matmul(Ub, Ua, D);   // ops[j] acts after ops[i]
          if (!A.mag.empty()) {
            const std::vector<double> Ma = embed(A.mag, A.qubits, {}, uni);
            const std::vector<double> Mb = embed(ops[j].mag, ops[j].qubits, {}, uni);
            A.mag = matmul(Mb, Ma, D);
          }
          A.qubits = uni;
          A.diag = is_diagonal(A.U, (int)uni.size());
          alive[j] = 0;
          break;
        }
        if (ti & tj) break;   // ops[j] cannot move past a block on its qubits
      }
    }
    for (size_t k = 0; k < ops.size(); k++)
      if (alive[k]) out.push_back(std::move(ops[k]));
  }
  return out;
}

// An op of site_blocks under construction.
namespace {
struct SiteOp {
  Block b;
  uint64_t touched_post = 0;   // qubits of moves after the sites
  uint64_t has_site = 0;
};
// Append "member y of the gate's qubits goes to perm[y]" to a table over the
// op's qubits.
void append_move(uint8_t *tab, const std::vector<int> &opq, const std::vector<int> &Q, const int *perm) {
  for (int y = 0; y < 8; y++) {
    const int v = tab[y];
    int c = 0;
    for (size_t j = 0; j < Q.size(); j++) c |= ((v >> index_of(opq, Q[j])) & 1) << j;
    const int r = perm[c];
    int w = v;
    for (size_t j = 0; j < Q.size(); j++) {
      const int bit = 1 << index_of(opq, Q[j]);
      w = ((r >> j) & 1) ? (w | bit) : (w & ~bit);
    }
    tab[y] = (uint8_t)w;
  }
}
}  // namespace

std::vector<Block> site_blocks(const std::vector<Gate> &gates, int K, std::vector<AdjSite> &sites) {
  std::vector<SiteOp> ops;
  std::vector<int> last(64, -1);
  std::vector<std::vector<int>> waiting(64);   // parametric gates not placed yet, by qubit
  auto is_sites = [&](int o) { return o >= 0 && ops[o].b.kind == TOP_SITES; };
  // give qubit q (of op o) its waiting gates as a site; o's sites on q come
  // before any move after the sites
  auto place = [&](int o, int q) {
    if (waiting[q].empty()) return;
    Block &b = ops[o].b;
    int &s = b.site[index_of(b.qubits, q)];
    if (s < 0) {
      s = (int)sites.size();
      sites.emplace_back();
    }
    sites[s].insert(sites[s].end(), waiting[q].begin(), waiting[q].end());
    waiting[q].clear();
    ops[o].has_site |= 1ull << q;
    last[q] = std::max(last[q], o);
  };
  auto new_op = [&]() {
    SiteOp n;
    n.b.kind = TOP_SITES;
    n.b.fusable = false;
    ops.push_back(std::move(n));
    return (int)ops.size() - 1;
  };
  // waiting gates of q that can only go to an op of their own (with other
  // qubits' waiting gates, neighbours first)
  auto place_alone = [&](int q) {
    if (waiting[q].empty()) return;
    if (is_sites(last[q]) && !((ops[last[q]].touched_post >> q) & 1)) return place(last[q], q);
    const int o = new_op();
    for (int d = 0; d < 64 && ops[o].b.qubits.size() < 3; d++)
      for (int x : {q + d, q - d}) {
        if (x < 0 || x >= 64 || waiting[x].empty() || ops[o].b.qubits.size() >= 3) continue;
        ops[o].b.qubits.push_back(x);
        place(o, x);
      }
  };
  for (const Gate &g : gates) {
    std::vector<int> Q = g.targets;
    Q.insert(Q.end(), g.controls.begin(), g.controls.end());
    if (g.inst >= 0) {
      const int q = Q[0], o = last[q];
      waiting[q].push_back(g.inst);
      // at once if the last op on q takes it; else with the next gate on q
      if (is_sites(o) && !((ops[o].touched_post >> q) & 1)) place(o, q);
      continue;
    }
    int perm[64];
    std::vector<cd> E;
    const bool narrow = Q.size() <= 3;
    if (narrow) E = embed(g.U, g.targets, g.controls, Q);
    if (narrow && permutation_of(E, (int)Q.size(), perm)) {
      int o = -1;
      for (int q : Q) o = std::max(o, last[q]);
      bool join = is_sites(o);
      if (join) {
        std::vector<int> uni = ops[o].b.qubits;
        for (int q : Q)
          if (index_of(uni, q) < 0) uni.push_back(q);
        join = uni.size() <= 3;
        // a qubit with gates waiting behind a move of this op needs another op
        for (int q : Q) join = join && (waiting[q].empty() || !((ops[o].touched_post >> q) & 1));
        if (join) ops[o].b.qubits = uni;
      }
      if (!join) {
        o = new_op();
        ops[o].b.qubits = Q;
      }
      for (int q : Q) place(o, q);
      const uint64_t m = qmask(Q);
      const bool pre = !(m & (ops[o].has_site | ops[o].touched_post));
      append_move(pre ? ops[o].b.pre : ops[o].b.post, ops[o].b.qubits, Q, perm);
      if (!pre) ops[o].touched_post |= m;
      for (int q : Q) last[q] = o;
      continue;
    }
    // a dense block, fused as in fuse()
    for (int q : Q) place_alone(q);
    int o = -1;
    for (int q : Q) o = std::max(o, last[q]);
    const bool alone = K <= 1 || g.controls.size() >= 2 || (int)Q.size() > K;
    if (!alone && o >= 0 && ops[o].b.kind == TOP_DENSE && ops[o].b.fusable) {
      Block &b = ops[o].b;
      std::vector<int> uni = b.qubits;
      for (int q : Q)
        if (index_of(uni, q) < 0) uni.push_back(q);
      if ((int)uni.size() <= K) {
        const std::vector<cd> Ub = embed(b.U, b.qubits, {}, uni);
        const std::vector<cd> Ug = embed(g.U, g.targets, g.controls, uni);
        b.U = matmul(Ug, Ub, 1 << (int)uni.size());
        b.qubits = uni;
        for (int q : uni) last[q] = std::max(last[q], o);
        continue;
      }
    }
    SiteOp n;
    if (alone) {
      n.b.qubits = g.targets;
      n.b.controls = g.controls;
      n.b.U = g.U;
      n.b.fusable = K > 1 && g.controls.empty();
    } else {
      n.b.qubits = Q;
      n.b.U = embed(g.U, g.targets, g.controls, Q);
    }
    ops.push_back(std::move(n));
    for (int q : Q) last[q] = (int)ops.size() - 1;
  }
  for (int q = 0; q < 64; q++) place_alone(q);
  std::vector<Block> out;
  out.reserve(ops.size());
  for (SiteOp &o : ops) {
    if (o.b.kind == TOP_DENSE) o.b.diag = is_diagonal(o.b.U, (int)o.b.qubits.size());
    out.push_back(std::move(o.b));
  }
  return out;
}

}  // namespace sv
