"""Gradient programs of sites (complex64) against the FP64 oracle's adjoint
gradient: every kind of gate, shared parameters, tile and batch sizes, and
passes beyond the kernel's op count."""
import numpy as np
import pytest

import workloads as W
from test_sites_cpu import mixed

pytestmark = pytest.mark.gpu


def check(oracle, c, p, terms, ev, g):
    """Probes and energies are FP32 products in short FP32 sums added in FP64:
    1e-5 of max(1, largest gradient), the bound of every gradient test."""
    ev_o, g_o, _ = oracle.adjoint_grad(c, p, terms)
    assert abs(ev - ev_o) <= 1e-5 * max(1, abs(ev_o), sum(abs(t[2]) for t in terms) * 0.1)
    assert np.max(np.abs(g - g_o)) <= 1e-5 * max(1, np.max(np.abs(g_o)))


def terms_of(n, rng):
    t = W.tfim(n) if n > 1 else [(1, 0, 0.5)]
    return t + [(1 << int(rng.integers(n)), int(rng.integers(1 << n)), float(rng.normal())) for _ in range(3)]


@pytest.mark.parametrize("n,m", [(5, 0), (6, 4), (8, 0), (10, 7), (11, 9), (13, 0), (13, 12), (14, 11)])
def test_mixed_circuits(svlib, oracle, n, m):
    rng = np.random.default_rng(10 * n + m)
    c = mixed(n, 80, n + m)
    # two gates of one parameter
    c.ops += [W.Op("RY", (0,), param=0), W.Op("RX", (n - 1,), param=0)]
    p = rng.uniform(-3, 3, c.n_params)
    terms = terms_of(n, rng)
    psi, lam = svlib.StateVector(n, "c64").set_basis(0), svlib.StateVector(n, "c64")
    ev, g = svlib.adjoint_grad(psi, lam, c, p, terms, opts=svlib.options(tile_m=m))
    check(oracle, c, p, terms, ev, g)
    back = psi.numpy()
    assert abs(abs(back[0]) - 1) <= 1e-5 and np.sum(np.abs(back[1:]) ** 2) <= 1e-9
    psi.close()
    lam.close()


@pytest.mark.parametrize("n,sets", [(3, 5), (4, 1), (9, 3), (12, 7), (16, 2), (17, 3)])
def test_ansatz_batches(svlib, oracle, n, sets):
    c = W.hea(n, 3)
    P = W.hea_params(sets, c.n_params, n)
    psi = [svlib.StateVector(n, "c64").set_basis(0) for _ in range(sets)]
    lam = [svlib.StateVector(n, "c64") for _ in range(sets)]
    ev, g = svlib.adjoint_grad_batch(psi, lam, c, P, W.tfim(n))
    for b in range(sets):
        check(oracle, c, P[b], W.tfim(n), ev[b], g[b])


def test_passes_beyond_the_op_count(svlib, oracle):
    """40 layers on 6 qubits: one tile takes them all, over 100 ops."""
    n = 6
    c = W.hea(n, 40)
    p = W.hea_params(1, c.n_params, 2)[0] * 0.2
    psi, lam = svlib.StateVector(n, "c64").set_basis(0), svlib.StateVector(n, "c64")
    ev, g = svlib.adjoint_grad(psi, lam, c, p, W.tfim(n))
    check(oracle, c, p, W.tfim(n), ev, g)


def test_energy_of_long_circuits(svlib, oracle):
    """The norm that FP32 rounding adds or takes is divided out: energies of 120
    layers within 2^-22 of the terms' weights (a sum of FP32 products in FP64;
    undivided, 1440 gates drift by several times that), over several seeds."""
    n, layers = 6, 120
    c = W.hea(n, layers)
    terms = W.tfim(n)
    psi, lam = svlib.StateVector(n, "c64"), svlib.StateVector(n, "c64")
    for seed in range(6):
        p = W.hea_params(1, c.n_params, seed)[0] * 0.1
        ev, g = svlib.adjoint_grad(psi.set_basis(0), lam, c, p, terms)
        ev_o, g_o, _ = oracle.adjoint_grad(c, p, terms)
        # the angles' matrices and 1440 gates' rounding turn the state as well:
        # a random walk of 2^-24 a gate
        tol = (2.0 ** -22 + 2.0 ** -24 * np.sqrt(2 * c.n_params)) * sum(abs(t[2]) for t in terms)
        assert abs(ev - ev_o) <= tol
    # a state the handle does not know is not taken for a unit vector
    half = np.zeros(1 << n, dtype=np.complex64)
    half[0] = 0.5
    ev4, g4 = svlib.adjoint_grad(psi.load(half), lam, c, p, terms)
    assert abs(4 * ev4 - ev) <= 1e-4 * abs(ev) and np.max(np.abs(4 * g4 - g)) <= 1e-4 * max(1, np.max(np.abs(g)))


def test_more_accumulators_than_15_bits(svlib):
    """22800 parameters, 34200 probe components: the energy's accumulator lies
    behind them (complex128, whose probes are one per parameter, as reference;
    FP32 rounding of 22800 gates grows as a random walk to 1e-5)."""
    n = 6
    c = W.hea(n, 1900)
    p = W.hea_params(1, c.n_params, 3)[0] * 0.05
    out = []
    for dt in ("c64", "c128"):
        psi, lam = svlib.StateVector(n, dt).set_basis(0), svlib.StateVector(n, dt)
        out.append(svlib.adjoint_grad(psi, lam, c, p, W.tfim(n)))
        psi.close()
        lam.close()
    (e0, g0), (e1, g1) = out
    assert abs(e0 - e1) <= 1e-3 and np.max(np.abs(g0 - g1)) <= 1e-3
