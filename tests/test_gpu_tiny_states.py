"""States of one to five qubits in every default plan, against the oracle."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("dt", ["c64", "c128"])
def test_circuits(svlib, oracle, dt, n):
    """40 layers, at most 60 roundings each way an amplitude: 2e-5 (complex64) and
    1e-13 (complex128) of the largest amplitude."""
    c = W.random_u3_cz(n, 40, n)
    s = svlib.StateVector(n, dt).set_basis(0).apply_circuit(c)
    want = oracle.run(c)
    assert np.max(np.abs(s.numpy() - want)) <= (2e-5 if dt == "c64" else 1e-13) * np.max(np.abs(want))
    s.close()
