// Host interpreter of the blocks gradient programs are made of (test only):
// site_blocks of a circuit, or of its reversed adjoint, applied to a state in
// complex128.
#include <complex>
#include <cstdio>
#include <vector>

#include "../../paper_2106_13995_gb300/csrc/sv_internal.h"

using namespace sv;

static void apply(std::vector<cd> &psi, const std::vector<int> &t, const std::vector<int> &ctl, const cd *U) {
  const int k = (int)t.size(), d = 1 << k;
  uint64_t tm = 0, cm = 0;
  for (int q : t) tm |= 1ull << q;
  for (int q : ctl) cm |= 1ull << q;
  std::vector<cd> x(d);
  for (uint64_t b = 0; b < psi.size(); b++) {
    if ((b & tm) || (b & cm) != cm) continue;
    auto at = [&](int y) {
      uint64_t i = b;
      for (int j = 0; j < k; j++) i |= (uint64_t)((y >> j) & 1) << t[j];
      return i;
    };
    for (int y = 0; y < d; y++) x[y] = psi[at(y)];
    for (int r = 0; r < d; r++) {
      cd a = 0;
      for (int y = 0; y < d; y++) a += U[r * d + y] * x[y];
      psi[at(r)] = a;
    }
  }
}
static void moves(std::vector<cd> &psi, const std::vector<int> &t, const uint8_t *to) {
  const int d = 1 << (int)t.size();
  std::vector<cd> U((size_t)d * d, 0.0);
  for (int y = 0; y < d; y++) U[(size_t)to[y] * d + y] = 1.0;
  apply(psi, t, {}, U.data());
}

// Applies the circuit (reverse: its adjoint) to psi; returns the number of
// blocks, *n_sites the number of sites, or -1.
extern "C" int sites_run(const sv_circuit *c, const double *params, double *psi_, int reverse, int K, int *n_sites) {
  const int n = c->n_qubits;
  std::vector<Gate> gates;
  if (circuit_to_gates(c, params, n, gates, true) != SV_OK) return -1;
  std::vector<std::vector<cd>> inst;
  for (Gate &g : gates)
    if (g.param >= 0) {
      g.inst = (int)inst.size();
      inst.push_back(reverse ? adjoint_of(g.U, 1) : g.U);
    }
  if (reverse) {
    gates = std::vector<Gate>(gates.rbegin(), gates.rend());
    for (Gate &g : gates) g.U = adjoint_of(g.U, (int)g.targets.size());
  }
  std::vector<AdjSite> sites;
  const std::vector<Block> blocks = site_blocks(gates, K, sites);
  *n_sites = (int)sites.size();
  cd *p = reinterpret_cast<cd *>(psi_);
  std::vector<cd> psi(p, p + (1ull << n));
  size_t seen = 0;
  for (const Block &b : blocks) {
    if (b.kind != TOP_SITES) {
      apply(psi, b.qubits, b.controls, b.U.data());
      continue;
    }
    if (b.qubits.empty() || b.qubits.size() > 3) return -1;
    moves(psi, b.qubits, b.pre);
    for (size_t j = 0; j < b.qubits.size(); j++) {
      if (b.site[j] < 0) continue;
      for (int i : sites[b.site[j]]) {
        apply(psi, {b.qubits[j]}, {}, inst[i].data());
        seen++;
      }
    }
    moves(psi, b.qubits, b.post);
  }
  if (seen != inst.size()) {
    std::printf("%zu of %zu parametric gates placed\n", seen, inst.size());
    return -1;
  }
  std::copy(psi.begin(), psi.end(), p);
  return (int)blocks.size();
}
