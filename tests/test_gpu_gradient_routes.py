"""Gradients whose fixed gates decide between sites and single gates, against
the FP64 oracle's."""
import numpy as np
import pytest

import workloads as W
from test_programs_cpu import ansatz

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,layers", [(6, 3), (12, 4), (16, 3)])
@pytest.mark.parametrize("route", ["H and CNOT", "CZ bricks", "CZ and CNOT"])
def test_routes(svlib, oracle, n, layers, route):
    """1e-5 of max(1, largest gradient), the bound of every gradient test."""
    c = ansatz(n, layers, {
        "H and CNOT": lambda k: [W.Op("X", (q + 1,), (q,)) for q in range(n - 1)],
        "CZ bricks": lambda k: [W.Op("CZ", (q, q + 1)) for q in range(k % 2, n - 1, 2)],
        "CZ and CNOT": lambda k: [W.Op("X", (q + 1,), (q,)) for q in range(n - 1)] + [W.Op("CZ", (0, n - 1))],
    }[route], ("H",) if route == "H and CNOT" else ())
    terms, sets = W.tfim(n), 3
    P = np.random.default_rng(n).uniform(-1, 1, (sets, c.n_params))
    psi = [svlib.StateVector(n, "c64").set_basis(0) for _ in range(sets)]
    lam = [svlib.StateVector(n, "c64") for _ in range(sets)]
    ev, g = svlib.adjoint_grad_batch(psi, lam, c, P, terms)
    for b in range(sets):
        ev_o, g_o, _ = oracle.adjoint_grad(c, P[b], terms)
        assert abs(ev[b] - ev_o) <= 1e-5 * max(1, abs(ev_o))
        assert np.max(np.abs(g[b] - g_o)) <= 1e-5 * max(1, np.max(np.abs(g_o)))
    for s in psi + lam:
        s.close()


@pytest.mark.parametrize("fixed", [(), ("H",)])
@pytest.mark.parametrize("n", [2, 8, 14])
def test_a_state_of_any_norm(svlib, oracle, n, fixed):
    """E = <psi_out|H|psi_out> of what the buffer holds, also where the caller
    wrote it after sv_set_basis: 0.81 of the unit vector's, within FP32
    rounding of the terms."""
    c = ansatz(n, 3, lambda k: [W.Op("X", (q + 1,), (q,)) for q in range(n - 1)], fixed)
    terms = W.tfim(n)
    p = np.random.default_rng(n).uniform(-1, 1, c.n_params)
    psi, lam = svlib.StateVector(n, "c64").set_basis(0), svlib.StateVector(n, "c64")
    psi.amps.mul_(0.9)
    ev, g = svlib.adjoint_grad(psi, lam, c, p, terms)
    ev_o, g_o, _ = oracle.adjoint_grad(c, p, terms)
    assert abs(ev - 0.81 * ev_o) <= 1e-5 * max(1, abs(ev_o))
    assert np.max(np.abs(g - 0.81 * g_o)) <= 1e-5 * max(1, np.max(np.abs(g_o)))


@pytest.mark.parametrize("scale", [0.75, 1.0 + 2.0 ** -8, 1.0 + 2.0 ** -12])
def test_a_matrix_that_is_not_unitary(svlib, oracle, scale):
    """Its factor stays in the energy, large or small, as in complex128."""
    n = 8
    c = ansatz(n, 2, lambda k: [W.Op("X", (q + 1,), (q,)) for q in range(n - 1)])
    c.ops.append(W.Op("MATRIX", (3,), matrix=scale * W.random_unitary(1, np.random.default_rng(1))))
    terms = W.tfim(n)
    p = np.random.default_rng(2).uniform(-1, 1, c.n_params)
    out = []
    for dt in ("c64", "c128"):
        psi, lam = svlib.StateVector(n, dt).set_basis(0), svlib.StateVector(n, dt)
        out.append(svlib.adjoint_grad(psi, lam, c, p, terms))
        psi.close()
        lam.close()
    (e0, g0), (e1, g1) = out
    assert abs(e1 - oracle.expect(oracle.run(c, params=p), terms)) <= 1e-12 * max(1, abs(e1))
    assert abs(e0 - e1) <= 1e-5 * max(1, abs(e1)) and np.max(np.abs(g0 - g1)) <= 1e-5 * max(1, np.max(np.abs(g1)))
