"""Small states whose circuits are planned in tiles of two sizes, against the
FP64 oracle."""
import numpy as np
import pytest

import workloads as W
from test_programs_cpu import toffolis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 12, 13, 14, 16, 18])
@pytest.mark.parametrize("dt", ["c64", "c128"])
def test_runs_alone_and_between_dense_gates(svlib, oracle, dt, n):
    """A run moves amplitudes exactly; with Hadamards around it, the bounds of
    the circuit tests (1e-5 and 1e-13 of the largest amplitude)."""
    rng = np.random.default_rng(n)
    run = toffolis(n, 300, rng)
    psi = W.random_state(n, rng).astype(np.complex64).astype(complex)
    s = svlib.StateVector(n, dt)
    c = W.Circuit(n, run)
    assert np.array_equal(s.load(psi).apply_circuit(c).numpy(), oracle.run(c, psi))
    h = W.hadamard_all(n).ops
    c = W.Circuit(n, h + run + h)
    want = oracle.run(c, psi)
    err = np.max(np.abs(s.load(psi).apply_circuit(c).numpy() - want)) / np.max(np.abs(want))
    assert err <= (1e-5 if dt == "c64" else 1e-13)
    s.close()


@pytest.mark.parametrize("n", [16, 17, 18])
def test_wide_blocks(svlib, oracle, n):
    c = W.block_chain(n, 6, n)
    psi = W.random_state(n, np.random.default_rng(n))
    s = svlib.StateVector(n, "c128")
    want = oracle.run(c, psi)
    assert np.max(np.abs(s.load(psi).apply_circuit(c).numpy() - want)) <= 1e-13 * np.max(np.abs(want))
    s.close()


@pytest.mark.parametrize("n", [18, 19, 20, 21])
@pytest.mark.parametrize("dt", ["c64", "c128"])
def test_tiles_from_one_to_many_per_sm(svlib, oracle, dt, n):
    """Passes whose CTAs are held to their share of each SM, twice in a row."""
    c = W.random_u3_cz(n, 3, n)
    s = svlib.StateVector(n, dt).set_basis(0).apply_circuit(c).apply_circuit(c)
    want = oracle.run(c, oracle.run(c))
    assert np.max(np.abs(s.numpy() - want)) <= (1e-5 if dt == "c64" else 1e-13) * np.max(np.abs(want))
    s.close()
