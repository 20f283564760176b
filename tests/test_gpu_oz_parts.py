"""Single amplitudes of complex128 circuits, small beside large ones, within
FP64 rounding of what the gates add up for each of them."""
import numpy as np
import pytest

import oz_cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [12, 14, 16])
@pytest.mark.parametrize("name", list(oz_cases.circuits(14, 0)))
def test_small_amplitudes_keep_their_digits(svlib, oracle, n, name):
    c = oz_cases.circuits(n, 0)[name]
    s = svlib.StateVector(n, "c128")
    for psi0 in oz_cases.states(n, n):
        oz_cases.check(oracle, c, psi0, s.load(psi0).apply_circuit(c).numpy(), name)
    s.close()


def test_parts_without_a_number(svlib):
    """A NaN or an infinity stays in its part: two settings of an idle qubit."""
    import workloads as W
    n = 14
    rng = np.random.default_rng(4)
    c = W.Circuit(n, [W.Op("RY", (3,), angles=(0.9,))])
    z = W.random_state(n, rng)
    s = svlib.StateVector(n, "c128")
    want = s.load(z).apply_circuit(c).numpy()
    for bad in (np.nan, np.inf):
        y = z.copy()
        y[5] = bad
        got = s.load(y).apply_circuit(c).numpy()
        hit = np.zeros(1 << n, dtype=bool)
        hit[[5, 5 ^ 8]] = True
        assert not np.any(np.isfinite(got[hit])) and np.array_equal(got[~hit], want[~hit])
    s.close()
