"""States whose width changes the default tile size, fusion width, threads per
tile or parameter-block size, against the FP64 oracle."""
import numpy as np
import pytest

import workloads as W
from conftest import fidelity_metrics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [2, 4, 7, 8, 10, 11, 12, 14, 17, 18, 19, 20, 21])
def test_default_plan_of_every_width(svlib, oracle, dt, n):
    """Mixed gates on a random state at both sides of each line.  Every gate
    rounds an amplitude a few times relative to the amplitudes it mixes, and
    the errors add like a random walk: 16 sqrt(gates) units of the largest
    amplitude bound them."""
    c = W.random_gate_circuit(n, 60, seed=n, kmax=min(3, n), cmax=2)
    psi0 = W.random_state(n, np.random.default_rng(n))
    s = svlib.StateVector(n, dt).load(psi0)
    want = oracle.run(c, s.numpy().astype(np.complex128))
    _, amp = fidelity_metrics(want, s.apply_circuit(c).numpy())
    eps = 2.0 ** -24 if dt == "c64" else 2.0 ** -53
    assert amp <= 16 * np.sqrt(len(c.ops)) * eps * np.max(np.abs(want)), amp
    s.close()


@pytest.mark.parametrize("nops", [10, 12, 13, 20, 24, 25])
def test_parameter_block_sizes(svlib, oracle, nops):
    """One pass of 3-qubit blocks at the ends of the small and middle parameter
    blocks (12 and 24 ops, 640 and 1280 matrix entries)."""
    n = 11
    rng = np.random.default_rng(nops)
    c = W.Circuit(n)
    for _ in range(nops):
        t = tuple(int(x) for x in rng.choice(n, size=3, replace=False))
        c.ops.append(W.Op("MATRIX", t, matrix=W.random_unitary(3, rng)))
    s = svlib.StateVector(n, "c64").set_basis(0)
    o = svlib.options(fusion_k=1, tile_m=n)
    want = oracle.run(c)
    _, amp = fidelity_metrics(want, s.apply_circuit(c, opts=o).numpy())
    assert amp <= 16 * np.sqrt(nops) * 2.0 ** -24 * np.max(np.abs(want)), amp
    s.close()
