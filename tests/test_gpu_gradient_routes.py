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
