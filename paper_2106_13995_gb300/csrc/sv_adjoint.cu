// C ABI: adjoint-method gradients (plain and batched) and batched circuit
// application.
//
// One "adjoint program" is a single list of tile passes:
//   forward   : the circuit on psi (1 vector per tile);
//   lambda    : lambda = H psi from Pauli strings, <H> = Re<psi|lambda>
//               (2 vectors: psi read-only, lambda written);
//   reverse   : for j = G..1, Im<lambda|G_j|psi> for parametric gates, then
//               U_j^dagger on both vectors (2 vectors).
// Parametric gates are kept as separate ops whose 2x2 matrices come from a
// per-batch table (forward U(theta_b) and reverse U(theta_b)^dagger), so one
// program serves every parameter set; fixed gates are fused as usual.  The
// batched form launches each pass once for all B states (grid.y = B).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>

#include "sv_internal.h"

namespace sv {

struct AdjointProgram {
  uint64_t serial = 0;            // unique per built program (graph cache key)
  DeviceProgram prog;
  std::vector<uint32_t> op0s;
  std::vector<int> inst_param;   // parameter index of each parametric instance
  std::vector<int> inst_gate;    // sv_gate of each parametric instance
  int n_params = 0;
  int n_inst = 0;
  // programs of sites (see site_blocks): the sites of both sweeps, and each
  // reverse site's first accumulator and components (bits: X, Y, Z);
  // without them one matrix per instance and one accumulator per parameter
  bool sites = false;
  bool split = false;            // some pass of sites was cut at other ops
  int folded = 0;                // gates that sites take: 4 per parametric gate, 3 per permutation
  std::vector<AdjSite> fwd_sites, rev_sites;
  std::vector<int> rev_slot, rev_comps;
  int n_acc = 0;                 // accumulators of the probes; TOP_DOT's follow
  bool norms = false;            // TOP_DOT takes <psi|psi> and Im <psi|lambda> too, <psi_in|psi_in> behind them
  bool unitary = false;          // every matrix op within kUnitaryTol
  int n_mats = 0;                // per-batch 2 x 2 matrices
};

static ProgCache<AdjointProgram> g_adj_cache(64);

// Recorded launch sequences of batched gradients (SV_MODE_TILED_GRAPH): the
// accumulator reset and every pass, per (first state, program, batch layout).
struct AdjGraph {
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};
using AdjGraphKey = std::pair<const sv_state *, std::vector<uint64_t>>;
static std::map<AdjGraphKey, AdjGraph> g_adj_graphs;
static std::mutex g_adj_graphs_mu;
constexpr size_t kMaxAdjGraphs = 32;

static void destroy_graph(AdjGraph &g) {
  if (g.exec) cudaGraphExecDestroy(g.exec);
  if (g.graph) cudaGraphDestroy(g.graph);
}

void drop_adjoint_programs(const sv_state *s) {
  g_adj_cache.drop_owner(s);
  std::lock_guard<std::mutex> lk(g_adj_graphs_mu);
  for (auto it = g_adj_graphs.begin(); it != g_adj_graphs.end();) {
    if (it->first.first == s) {
      destroy_graph(it->second);
      it = g_adj_graphs.erase(it);
    } else {
      ++it;
    }
  }
}

// Passes of TOP_SITES ops have a kernel of their own: split a pass where it
// changes between them and other ops, and beyond the kernel's op count.
static std::vector<PassPlan> split_sites(const std::vector<PassPlan> &passes, bool &split) {
  std::vector<PassPlan> out;
  for (const PassPlan &P : passes) {
    size_t i = 0;
    do {
      PassPlan Q;
      Q.S = P.S;
      const bool sites = i < P.ops.size() && P.ops[i].kind == TOP_SITES;
      while (i < P.ops.size() && (P.ops[i].kind == TOP_SITES) == sites &&
             (!sites || Q.ops.size() < (size_t)kMaxSitesOps))
        Q.ops.push_back(P.ops[i++]);
      split = split || (i < P.ops.size() && (P.ops[i].kind == TOP_SITES) != sites);
      out.push_back(std::move(Q));
    } while (i < P.ops.size());
  }
  return out;
}

static void append_passes(DeviceProgram &prog, std::vector<uint32_t> &op0s, const std::vector<PassPlan> &passes,
                          const BuildCtx &b, const std::vector<int> &bmo, sv_status &st) {
  for (const PassPlan &P : passes) {
    if (st != SV_OK) return;
    st = emit_pass(prog, P, b, op0s, bmo);
  }
}

static sv_status build_adjoint(sv_state *s, const sv_circuit *c, const double *params0,
                               const sv_pauli_term *terms, int nt, const Opts &o1, const Opts &o2, bool sites,
                               bool norms, AdjointProgram &A) {
  std::vector<Gate> gates;
  SV_TRY(circuit_to_gates(c, params0, s->n, gates, true));
  A.n_params = c->n_params;
  for (Gate &g : gates) {
    if (g.param < 0) continue;
    if (g.targets.size() != 1 || !g.controls.empty() || gate_generator(g.param_gate) == 0)
      return set_error(SV_EUNSUPPORTED,
                       "parametric gates must be uncontrolled single-qubit RX/RY/RZ/PHASE for gradients");
    g.inst = A.n_inst++;
    A.inst_param.push_back(g.param);
    A.inst_gate.push_back(g.param_gate);
  }
  const int G = (int)gates.size();
  // The reverse sweep of a matrix op that is not unitary undoes nothing; what a
  // probe and an adjoint per gate add up then is kept as it is.  Up to FP32
  // rounding an op passes for unitary.
  double off = 0;
  for (int i = 0; i < G; i++)
    if (c->ops[i].gate == SV_GATE_MATRIX) {
      const double e = unitarity_error(gates[i].U, (int)gates[i].targets.size());
      off = e <= off ? off : e;   // (a NaN stays)
    }
  A.unitary = off <= kUnitaryTol;
  if (!(off <= 1e-6)) sites = norms = false;
  int perm[64];
  for (const Gate &g : gates)
    if (g.inst >= 0) A.folded += 4;
    else if (g.targets.size() + g.controls.size() <= 3 && permutation_of(g.U, (int)g.targets.size(), perm)) A.folded += 3;
  A.sites = sites;
  A.norms = norms;
  A.n_acc = A.n_params;
  A.n_mats = 2 * A.n_inst;
  std::vector<Block> fwd_blocks, rev_blocks;
  std::vector<int> fwd_mat, rev_mat;
  if (sites) {
    fwd_blocks = site_blocks(gates, o1.fusion_k, A.fwd_sites);
    std::vector<Gate> rev(gates.rbegin(), gates.rend());
    for (Gate &g : rev) g.U = adjoint_of(g.U, (int)g.targets.size());
    rev_blocks = site_blocks(rev, o2.fusion_k, A.rev_sites);
    A.n_acc = 0;
    for (const AdjSite &st : A.rev_sites) {
      int c = 0;
      for (int i : st) c |= 1 << (std::min(3, gate_generator(A.inst_gate[i])) - 1);
      if (st.size() > 1) c |= 7;   // later gates' generators turn into the other two
      A.rev_slot.push_back(A.n_acc);
      A.rev_comps.push_back(c);
      A.n_acc += __builtin_popcount(c);
    }
    for (size_t i = 0; i < A.fwd_sites.size(); i++) fwd_mat.push_back(4 * (int)i);
    for (size_t i = 0; i < A.rev_sites.size(); i++) rev_mat.push_back(4 * (int)(A.fwd_sites.size() + i));
    A.n_mats = (int)(A.fwd_sites.size() + A.rev_sites.size());
  }
  std::vector<int> fwd_off(A.n_inst), rev_off(A.n_inst);
  for (int i = 0; i < A.n_inst; i++) {
    fwd_off[i] = 4 * i;
    rev_off[i] = 4 * (A.n_inst + i);
  }
  sv_status st = SV_OK;
  // forward
  {
    std::vector<Block> blocks = sites ? std::move(fwd_blocks) : fuse(gates, o1.fusion_k);
    int m = o1.tile_m, L = o1.L;
    if (!fit_tile(blocks, s->n, lmin(s->dt), mmax(s->dt, 1), m, L))
      return set_error(SV_EUNSUPPORTED, "a fused block does not fit a shared-memory tile");
    std::vector<PassPlan> passes = plan_passes(blocks, s->n, m, L, 256, 1 << 16);
    if (passes.empty() && !blocks.empty()) return set_error(SV_EINVAL, "internal: pass planning failed");
    BuildCtx b{s->dt, s->n, m, L, 1, 0};
    b.site_mat = fwd_mat.data();
    append_passes(A.prog, A.op0s, split_sites(passes, A.split), b, fwd_off, st);
    // (gather tables in front move the amplitudes and leave the norm)
    for (size_t i = 0; norms && st == SV_OK && i < A.prog.passes.size(); i++)
      if (!(A.prog.passes[i].flags & kPassTable)) {
        A.prog.passes[i].flags |= kPassNorm;
        A.prog.passes[i].mat0 = (uint32_t)A.n_acc + 3;
        break;
      }
  }
  // lambda = H psi
  {
    std::vector<Block> blocks;
    for (int t = 0; t < nt; t++) {
      Block b;
      b.kind = TOP_PAULI;
      for (int q = 0; q < s->n; q++)
        if ((terms[t].x_mask >> q) & 1) b.qubits.push_back(q);
      b.xmask = terms[t].x_mask;
      b.zmask = terms[t].z_mask;
      b.coeff = terms[t].coeff;
      b.fusable = false;
      blocks.push_back(b);
    }
    int m = o2.tile_m, L = o2.L;
    if (!fit_tile(blocks, s->n, lmin(s->dt), mmax(s->dt, 2), m, L))
      return set_error(SV_EUNSUPPORTED, "a Pauli string's X support does not fit a shared-memory tile");
    std::vector<PassPlan> passes = plan_passes(blocks, s->n, m, L, 256, 1 << 16);
    if (passes.empty() && !blocks.empty()) return set_error(SV_EINVAL, "internal: pass planning failed");
    if (passes.empty()) {
      PassPlan P;
      for (int q = 0; q < std::min(m, s->n); q++) P.S.push_back(q);
      passes.push_back(P);
    }
    Block zero;
    zero.kind = TOP_ZERO;
    passes.front().ops.insert(passes.front().ops.begin(), zero);
    Block dot;
    dot.kind = TOP_DOT;
    dot.slot = A.n_acc;
    dot.gen = norms;
    passes.back().ops.push_back(dot);
    for (size_t i = 0; i < passes.size() && st == SV_OK; i++) {
      BuildCtx b{s->dt, s->n, m, L, 2, (i == 0 ? 1u : 0u) | 2u};
      st = emit_pass(A.prog, passes[i], b, A.op0s, {});
    }
  }
  // reverse sweep
  {
    std::vector<Gate> rev;
    rev.reserve(2 * G);
    for (int j = G - 1; j >= 0 && !sites; j--) {
      const Gate &g = gates[j];
      if (g.param >= 0) {
        Gate probe;
        probe.targets = g.targets;
        probe.grad_gen = gate_generator(g.param_gate);
        probe.grad_slot = g.param;
        rev.push_back(probe);
      }
      Gate u = g;
      u.U = adjoint_of(g.U, (int)g.targets.size());
      rev.push_back(u);
    }
    std::vector<Block> blocks = sites ? std::move(rev_blocks) : fuse(rev, o2.fusion_k);
    for (Block &b : blocks)
      if (b.kind == TOP_DENSE || b.kind == TOP_SITES) b.vmask = 3;
    int m = o2.tile_m, L = o2.L;
    if (!fit_tile(blocks, s->n, lmin(s->dt), mmax(s->dt, 2), m, L))
      return set_error(SV_EUNSUPPORTED, "a fused block does not fit a shared-memory tile");
    std::vector<PassPlan> passes = plan_passes(blocks, s->n, m, L, 256, 1 << 16);
    if (passes.empty() && !blocks.empty()) return set_error(SV_EINVAL, "internal: pass planning failed");
    BuildCtx b{s->dt, s->n, m, L, 2, 0};
    b.site_mat = rev_mat.data();
    b.site_slot = A.rev_slot.data();
    b.site_comps = A.rev_comps.data();
    const size_t first = A.prog.passes.size();
    append_passes(A.prog, A.op0s, split_sites(passes, A.split), b, rev_off, st);
    if (sites && st == SV_OK && A.prog.passes.size() > first) {
      A.prog.passes[first].flags |= kPassShift;
      A.prog.passes[first].mat0 = (uint32_t)A.n_acc;
    }
  }
  return st;
}

// One matrix per site: the product of its gates' matrices (adjoints in the
// reverse sweep), in FP64.
static void put_site_mats(std::vector<uint8_t> &pool, const AdjointProgram &A, const double *theta) {
  std::vector<cd> U;
  for (int pass = 0; pass < 2; pass++)
    for (const AdjSite &st : pass == 0 ? A.fwd_sites : A.rev_sites) {
      cd M[4] = {1.0, 0.0, 0.0, 1.0};
      for (int i : st) {
        const double ang[3] = {theta[A.inst_param[i]], 0, 0};
        gate_matrix(A.inst_gate[i], ang, U);
        if (pass == 1) U = adjoint_of(U, 1);
        const cd N[4] = {U[0] * M[0] + U[1] * M[2], U[0] * M[1] + U[1] * M[3], U[2] * M[0] + U[3] * M[2],
                         U[2] * M[1] + U[3] * M[3]};
        std::memcpy(M, N, sizeof(M));
      }
      put_pairs_c64(pool, M, 1);
    }
}

// The gradients of a site from its components: p_G = Im <lambda| G |psi> at
// the run's start.  Undoing U = exp(-i theta P / 2) on both vectors turns p_G
// into Im <lambda| U G U^dagger |psi>, a rotation of (X, Y, Z) about P.
static void site_grads(const AdjointProgram &A, const double *theta, const double *acc, double *grad) {
  for (size_t k = 0; k < A.rev_sites.size(); k++) {
    double p[3] = {0, 0, 0};   // X, Y, Z
    int at = A.rev_slot[k];
    for (int g = 0; g < 3; g++)
      if ((A.rev_comps[k] >> g) & 1) p[g] = acc[at++];
    for (int i : A.rev_sites[k]) {
      const int gen = gate_generator(A.inst_gate[i]);
      // PHASE's generator diag(0, -2) is Z - I, and <lambda|psi> = <psi|H|psi>
      // has no imaginary part
      grad[A.inst_param[i]] += p[std::min(gen, 3) - 1];
      const double c = std::cos(theta[A.inst_param[i]]), s = std::sin(theta[A.inst_param[i]]);
      const double x = p[0], y = p[1], z = p[2];
      if (gen == 1) {
        p[1] = c * y + s * z;
        p[2] = c * z - s * y;
      } else if (gen == 2) {
        p[2] = c * z + s * x;
        p[0] = c * x - s * z;
      } else {
        p[0] = c * x + s * y;
        p[1] = c * y - s * x;
      }
    }
  }
}

template <typename R>
static void put_mats(std::vector<uint8_t> &pool, const AdjointProgram &A, const double *theta) {
  // forward matrices for every instance, then their adjoints
  std::vector<cd> U;
  for (int pass = 0; pass < 2; pass++)
    for (int i = 0; i < A.n_inst; i++) {
      const double ang[3] = {theta[A.inst_param[i]], 0, 0};
      gate_matrix(A.inst_gate[i], ang, U);
      if (pass == 1) U = adjoint_of(U, 1);
      if constexpr (sizeof(R) == 4) {
        put_pairs_c64(pool, U.data(), 1);   // the layout complex64 tile ops read
      } else {
        for (int e = 0; e < 4; e++) {
          R v[2] = {(R)U[e].real(), (R)U[e].imag()};
          const uint8_t *p = (const uint8_t *)v;
          pool.insert(pool.end(), p, p + sizeof(v));
        }
      }
    }
}

static sv_status check_batch(sv_state *const *psi, int B, int n, sv_dtype dt, cudaStream_t st) {
  for (int b = 0; b < B; b++) {
    if (!psi[b]) return set_error(SV_EINVAL, "null state in batch");
    if (psi[b]->n != n || psi[b]->dt != dt) return set_error(SV_EINVAL, "batch states differ in width or dtype");
    if (psi[b]->stream != st) return set_error(SV_EINVAL, "batch states must share one stream");
  }
  return SV_OK;
}

// The program of a circuit's gradient for B parameter sets, from the cache or
// built.  lean: the one that takes least of the workspace, a probe and a matrix
// per gate, one accumulator per parameter and one for the energy.
static sv_status adjoint_program(sv_state *s, const sv_circuit *c, const double *params, const sv_pauli_term *terms,
                                 int nt, const sv_options *opt, int B, bool lean,
                                 std::shared_ptr<const AdjointProgram> &Ap) {
  Opts o1 = resolve(s, opt, 1), o2 = resolve(s, opt, 2);
  // defaults for the gradient program (measured on the 20-qubit, 64-set
  // ansatz): fusion width 2 and 12-qubit tiles for both sweeps
  if (!opt || opt->fusion_k == 0) o1.fusion_k = o2.fusion_k = 2;
  if (!opt || opt->tile_m == 0) {
    // (12-qubit tiles; 10 for small states and few sets, whose tiles would
    // not fill the GPU: one set of 16 qubits 441 -> 329 us, of 18 qubits
    // 497 -> 398; at 20 qubits 700 -> 776)
    int lb = 0;
    while ((2 << lb) <= B) lb++;
    o1.tile_m = o2.tile_m = std::min(s->dt == SV_C64 && !lean && s->n + lb <= 18 ? 10 : 12, s->n);
    o1.L = o2.L = std::min(o1.L, o1.tile_m);
  }
  // cache key: circuit structure, terms, options (parameters enter only the
  // per-batch matrices, uploaded every call)
  KeyBytes k;
  k.val((int)0xad);
  SV_TRY(circuit_key(k, c, s->n));
  if (nt) k.bytes(terms, sizeof(sv_pauli_term) * nt);
  k.val(o1);
  k.val(o2);
  k.val(s->dt);
  // complex64 programs are made of sites; complex128 ones are bound by FP64
  // arithmetic, which the probes of three components a site would add to
  const bool sites = s->dt == SV_C64 && !lean && s->n >= 3 && o1.tile_m >= 3 && o2.tile_m >= 3;
  const bool norms = s->dt == SV_C64 && !lean;
  k.val((int)sites);
  k.val((int)norms);
  const uint64_t kh = k.hash();
  Ap = g_adj_cache.find(s, k, kh);
  if (!Ap) {
    auto built = std::make_shared<AdjointProgram>();
    SV_TRY(build_adjoint(s, c, params, terms, nt, o1, o2, sites, norms, *built));
    if (built->split) {
      // Fixed gates that are not permutations cut passes of sites; a launch
      // more, with its read and write of the vectors, costs what four
      // parametric or five permutation gates in sites save (ms
      // in sites and with a probe and a matrix per gate, six layers of RY and
      // RZ, 26 qubits: CNOT ladder, no cut 32.5 and 87, H before each RY 73 and
      // 91, one CZ a layer 41 and 92, CZ ladder 128 and 119, CZ bricks 112 and
      // 82, only the last layer parametric 58 and 49; 16 qubits 0.28 and 0.76,
      // 0.63 and 0.81, 0.37 and 0.80, 0.80 and 0.85, 0.73 and 0.65, 0.49 and
      // 0.45)
      auto plain = std::make_shared<AdjointProgram>();
      SV_TRY(build_adjoint(s, c, params, terms, nt, o1, o2, false, norms, *plain));
      const int more = (int)built->prog.passes.size() - (int)plain->prog.passes.size();
      if (16 * more > built->folded) built = std::move(plain);
    }
    built->serial = next_program_serial();
    Ap = g_adj_cache.insert(s, k, kh, std::move(built));
  }
  return SV_OK;
}

// Bytes of the workspace for B parameter sets.
static ProgLayout adjoint_layout(const sv_state *s, const AdjointProgram &A, int B) {
  return layout_of(A.prog, 2 * (size_t)B * sizeof(void *), (size_t)B * A.n_mats * 4 * amp_bytes(s->dt));
}
static size_t adjoint_acc_stride(const AdjointProgram &A) { return (size_t)A.n_acc + (A.norms ? 4 : 1); }

// The same, lean where the program would outgrow the workspace (a site takes
// 128 bytes a sweep on its own, a single gate 128 in all).
static sv_status fitting_program(sv_state *s, const sv_circuit *c, const double *params, const sv_pauli_term *terms,
                                 int nt, const sv_options *opt, int B, std::shared_ptr<const AdjointProgram> &Ap) {
  for (bool lean : {false, true}) {
    SV_TRY(adjoint_program(s, c, params, terms, nt, opt, B, lean, Ap));
    if (adjoint_layout(s, *Ap, B).end <= kWsProgBytes &&
        adjoint_acc_stride(*Ap) * B * sizeof(double) <= red_bytes(s->n))
      break;
  }
  return SV_OK;
}

sv_status adjoint_plan(sv_state *s, const sv_circuit *c, const double *params, const sv_pauli_term *terms, int nt,
                       const sv_options *opt, int B, AdjointPlan &out) {
  std::shared_ptr<const AdjointProgram> Ap;
  SV_TRY(fitting_program(s, c, params, terms, nt, opt, B, Ap));
  out.passes = (int)Ap->prog.passes.size();
  out.sites = Ap->sites;
  out.prog_bytes = adjoint_layout(s, *Ap, B).end;
  out.acc_bytes = adjoint_acc_stride(*Ap) * B * sizeof(double);
  return SV_OK;
}

static sv_status adjoint_batch(sv_state *const *psi, sv_state *const *lam, int B, const sv_circuit *c,
                               const double *params, const sv_pauli_term *terms, int nt, const sv_options *opt,
                               double *ev_out, double *grad_out) {
  if (!psi || !lam || B < 1 || !c || !ev_out || (c->n_params > 0 && (!params || !grad_out)))
    return set_error(SV_EINVAL, "null argument");
  sv_state *s = psi[0];
  if (!s) return set_error(SV_EINVAL, "null state");
  SV_TRY(check_batch(psi, B, s->n, s->dt, s->stream));
  SV_TRY(check_batch(lam, B, s->n, s->dt, s->stream));
  for (int b = 0; b < B; b++) psi[b]->basis_known = lam[b]->basis_known = false;
  if (nt < 0 || (nt > 0 && !terms)) return set_error(SV_EINVAL, "bad term list");
  const uint64_t lim = (1ull << s->n) - 1;
  for (int t = 0; t < nt; t++)
    if ((terms[t].x_mask & ~lim) || (terms[t].z_mask & ~lim))
      return set_error(SV_EINVAL, "Pauli mask references a qubit >= n");
  const int np = c->n_params;
  std::shared_ptr<const AdjointProgram> Ap;
  SV_TRY(fitting_program(s, c, params, terms, nt, opt, B, Ap));
  const AdjointProgram &A = *Ap;
  // per-batch matrices, state pointer tables
  std::vector<uint8_t> pm;
  pm.reserve((size_t)B * A.n_mats * 4 * (s->dt == SV_C64 ? 8 : 16));
  for (int b = 0; b < B; b++) {
    if (A.sites) put_site_mats(pm, A, params + (size_t)b * np);
    else if (s->dt == SV_C64) put_mats<float>(pm, A, params + (size_t)b * np);
    else put_mats<double>(pm, A, params + (size_t)b * np);
  }
  std::vector<void *> tbl(2 * (size_t)B);
  for (int b = 0; b < B; b++) {
    tbl[b] = psi[b]->amps;
    tbl[B + b] = lam[b]->amps;
  }
  const ProgLayout L = adjoint_layout(s, A, B);
  SV_TRY(stage_upload(s,
                      {{A.prog.ops.data(), A.prog.ops.size() * sizeof(TileOp)},
                       {A.prog.mats.data(), A.prog.mats.size()},
                       {A.prog.coeffs.data(), A.prog.coeffs.size() * sizeof(double)},
                       {tbl.data(), tbl.size() * sizeof(void *)},
                       {pm.data(), pm.size()}},
                      {L.ops_off, L.mats_off, L.coeffs_off, L.tbl_off, L.pmats_off}, L.end));
  const size_t acc_stride = adjoint_acc_stride(A);
  const size_t acc_bytes = acc_stride * B * sizeof(double);
  if (acc_bytes > red_bytes(s->n)) return set_error(SV_ENOMEM, "workspace too small for the gradient batch");
  double *acc = reinterpret_cast<double *>(s->ws + kWsRed);
  char *base = s->ws + kWsProg;
  LaunchEnv E;
  E.batch = B;
  E.tbl0 = reinterpret_cast<void *const *>(base + L.tbl_off);
  E.tbl1 = E.tbl0 + B;
  E.pmats = base + L.pmats_off;
  E.pmats_stride = (uint64_t)4 * A.n_mats;
  E.acc = acc;
  E.acc_stride = acc_stride;
  if (opt && opt->mode == SV_MODE_TILED_GRAPH) {
    // the reset and all passes as one recorded launch sequence; the tables
    // and per-set matrices were uploaded above, in stream order, so a
    // replay reads this call's parameters
    std::lock_guard<std::mutex> lk(g_adj_graphs_mu);
    AdjGraphKey gk{s, {Ap->serial, (uint64_t)B, (uint64_t)L.end, (uint64_t)acc_bytes}};
    auto it = g_adj_graphs.find(gk);
    if (it == g_adj_graphs.end()) {
      AdjGraph g;
      if (!s->capture) SV_CUDA(cudaStreamCreateWithFlags(&s->capture, cudaStreamNonBlocking));
      SV_CUDA(cudaStreamBeginCapture(s->capture, cudaStreamCaptureModeThreadLocal));
      cudaError_t e1 = cudaMemsetAsync(acc, 0, acc_bytes, s->capture);
      sv_status st = e1 == cudaSuccess ? launch_program(s, A.prog, L, A.op0s, E, s->capture)
                                       : cuda_error(e1, "cudaMemsetAsync");
      cudaError_t e2 = cudaStreamEndCapture(s->capture, &g.graph);
      if (st != SV_OK) {
        destroy_graph(g);
        return st;
      }
      if (e2 != cudaSuccess) return cuda_error(e2, "cudaStreamEndCapture");
      cudaError_t e3 = cudaGraphInstantiate(&g.exec, g.graph, 0);
      if (e3 != cudaSuccess) {
        destroy_graph(g);
        return cuda_error(e3, "cudaGraphInstantiate");
      }
      if (g_adj_graphs.size() >= kMaxAdjGraphs) {
        SV_CUDA(cudaStreamSynchronize(s->stream));   // replays in flight finish first
        for (auto &kv : g_adj_graphs) destroy_graph(kv.second);
        g_adj_graphs.clear();
      }
      it = g_adj_graphs.emplace(std::move(gk), g).first;
    }
    SV_CUDA(cudaGraphLaunch(it->second.exec, s->stream));
    g_launches++;
  } else {
    SV_CUDA(cudaMemsetAsync(acc, 0, acc_bytes, s->stream));
    SV_TRY(launch_program(s, A.prog, L, A.op0s, E));
  }
  std::vector<double> h(acc_stride * B);
  SV_CUDA(cudaMemcpyAsync(h.data(), acc, acc_bytes, cudaMemcpyDeviceToHost, s->stream));
  SV_CUDA(cudaStreamSynchronize(s->stream));
  for (int b = 0; b < B; b++) {
    const double *hb = h.data() + (size_t)b * acc_stride;
    ev_out[b] = hb[A.n_acc];
    if (A.sites) {
      std::fill(grad_out + (size_t)b * np, grad_out + (size_t)(b + 1) * np, 0.0);
      site_grads(A, params + (size_t)b * np, hb, grad_out + (size_t)b * np);
    } else {
      for (int p = 0; p < np; p++) grad_out[(size_t)b * np + p] = hb[p];
    }
    // A unitary circuit leaves the norm alone; what FP32 rounding made of it
    // (1e-6 after some hundred gates, the largest part of the energy's error) is
    // divided out.  A larger change is not rounding.
    if (A.norms && A.unitary) {
      const double drift = hb[A.n_acc + 1] / hb[A.n_acc + 3];
      if (std::fabs(drift - 1.0) < 1e-3) {
        ev_out[b] /= drift;
        for (int p = 0; p < np; p++) grad_out[(size_t)b * np + p] /= drift;
      }
    }
  }
  return SV_OK;
}

}  // namespace sv

using namespace sv;

extern "C" {

sv_status sv_adjoint_grad(sv_state *psi, sv_state *lam, const sv_circuit *c, const double *params,
                          const sv_pauli_term *terms, int nt, const sv_options *opt, double *ev, double *grad) {
  if (!psi || !lam) return set_error(SV_EINVAL, "null state");
  if (psi == lam || psi->amps == lam->amps) return set_error(SV_EINVAL, "psi and lambda must be distinct buffers");
  return adjoint_batch(&psi, &lam, 1, c, params, terms, nt, opt, ev, grad);
}

sv_status sv_adjoint_grad_batch(sv_state *const *psi, sv_state *const *lam, int B, const sv_circuit *c,
                                const double *params, const sv_pauli_term *terms, int nt, const sv_options *opt,
                                double *ev, double *grad) {
  return adjoint_batch(psi, lam, B, c, params, terms, nt, opt, ev, grad);
}

}  // extern "C"
