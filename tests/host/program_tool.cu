// Programs as the library builds them, on a host-only state (test only).
#include <cstring>

#include "../../paper_2106_13995_gb300/csrc/sv_internal.h"

using namespace sv;

static sv_state host_state(int n, int dt) {
  sv_state s;
  s.n = n;
  s.dt = (sv_dtype)dt;
  s.ws_bytes = sv_workspace_bytes(n, (sv_dtype)dt);
  return s;
}

// Build a circuit's program: returns the status, *end the bytes of the program
// area it takes, flags[0 .. *n_passes) each pass's flags (at most cap).
extern "C" int program_build(const sv_circuit *c, int dt, const sv_options *opt, uint64_t *end, uint32_t *flags, int cap,
                             int *n_passes) {
  sv_state s = host_state(c->n_qubits, dt);
  ProgramRef cp;
  Opts o;
  const sv_status st = get_program(&s, c, nullptr, opt, &cp, &o);
  if (st != SV_OK) return (int)st;
  *end = cp->lay.end;
  *n_passes = (int)cp->prog.passes.size();
  for (int i = 0; i < *n_passes && i < cap; i++) flags[i] = cp->prog.passes[i].flags;
  return SV_OK;
}

extern "C" uint64_t program_area() { return kWsProgBytes; }

// Passes a gradient of B parameter sets launches, *sites whether they are made of
// sites, *prog and *acc the bytes of the program and of the reduction area it
// takes; -status on an error.
extern "C" int gradient_passes(const sv_circuit *c, const double *params, const sv_pauli_term *terms, int nt, int B,
                               int dt, int *sites, uint64_t *prog, uint64_t *acc) {
  sv_state s = host_state(c->n_qubits, dt);
  AdjointPlan p;
  const sv_status st = adjoint_plan(&s, c, params, terms, nt, nullptr, B, p);
  *sites = p.sites;
  *prog = p.prog_bytes;
  *acc = p.acc_bytes;
  return st == SV_OK ? p.passes : -(int)st;
}

extern "C" uint64_t reduction_area(int n) { return red_bytes(n); }

// Options a circuit runs with after the autotuner's cache: fusion width, tile
// size, and whether the tensor-core and permutation paths are open.
extern "C" void tuned(const sv_circuit *c, int dt, int *out) {
  sv_state s = host_state(c->n_qubits, dt);
  Opts o = resolve(&s, nullptr, 1);
  tuned_options(&s, c, nullptr, o);
  out[0] = o.fusion_k;
  out[1] = o.tile_m;
  out[2] = o.oz;
  out[3] = o.moves;
}

// sv_plan_fmas on a host-only state
extern "C" double plan_fmas(const sv_circuit *c, int dt) {
  sv_state s = host_state(c->n_qubits, dt);
  double f = -1;
  return sv_plan_fmas(&s, c, nullptr, nullptr, &f) == SV_OK ? f : -1;
}

// |index> through the circuit op by op, as sv_apply_circuit follows a known
// basis state: 1 and the final index and amplitude, 0 when some gate does not
// keep a basis state, -status on an error.
extern "C" int follow_basis(const sv_circuit *c, const double *params, uint64_t index, uint64_t *out_index, double *amp) {
  cd a = 1.0;
  bool stays = false;
  const sv_status st = propagate_circuit(c, params, c->n_qubits, index, a, stays);
  if (st != SV_OK) return -(int)st;
  *out_index = index;
  amp[0] = a.real();
  amp[1] = a.imag();
  return stays;
}
