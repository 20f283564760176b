"""Single gates by 16-byte units: diagonal gates whose idle qubits are left out
and 1- and 2-qubit gates of two groups a unit, against the FP64 oracle."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def reference(psi, n, u, t, c):
    """U on targets t (bit j of a row <-> t[j]) where all controls are 1, in
    complex128."""
    idx = np.arange(1 << n)
    on = np.ones(1 << n, dtype=bool)
    for q in c:
        on &= ((idx >> q) & 1) == 1
    y = np.zeros_like(idx)
    base = idx.copy()
    for j, q in enumerate(t):
        y |= ((idx >> q) & 1) << j
        base &= ~(1 << q)
    out = np.zeros_like(psi)
    for col in range(1 << len(t)):
        src = base.copy()
        for j, q in enumerate(t):
            src |= ((col >> j) & 1) << q
        out += u[y, col] * psi[src]
    return np.where(on, out, psi)


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 11, 14])
def test_diagonal_gates(svlib, n, dt):
    """Idle targets, idle controls, none, all (the identity), with and without
    qubit 0; what is left out keeps its bits."""
    rng = np.random.default_rng(n)
    for trial in range(24):
        k = int(rng.integers(1, min(n, 3) + 1))
        nc = int(rng.integers(0, min(n - k, 3) + 1))
        q = [int(x) for x in rng.permutation(n)[:k + nc]]
        d = np.exp(2j * np.pi * rng.random(1 << k))
        keep = rng.integers(0, 4)
        if keep == 1:
            d[0] = 1
        elif keep == 2:
            d[:-1] = 1
        elif keep == 3 and trial % 2:
            d[:] = 1
        psi = W.random_state(n, rng).astype(np.complex64 if dt == "c64" else np.complex128)
        s = svlib.StateVector(n, dt).load(psi)
        s.apply_gate(np.diag(d), tuple(q[:k]), tuple(q[k:]))
        got, want = s.numpy(), reference(psi.astype(np.complex128), n, np.diag(d), q[:k], q[k:])
        # one complex product: 2 roundings of it and one of the phase
        assert np.max(np.abs(got - want)) <= 4 * np.finfo(got.real.dtype).eps * np.max(np.abs(psi))
        same = want == psi
        assert np.array_equal(got[same], psi[same])
        s.close()


@pytest.mark.parametrize("n", [2, 3, 4, 7, 12, 15])
def test_dense_gates_by_pairs(svlib, n):
    """1 to 3 targets (3: by single amplitudes), 0 to 3 controls, with and without qubit 0; permutation
    matrices move bits."""
    rng = np.random.default_rng(100 + n)
    for trial in range(24):
        k = int(rng.integers(1, min(n, 3) + 1))
        nc = int(rng.integers(0, min(n - k, 3) + 1))
        q = [int(x) for x in rng.permutation(n)[:k + nc]]
        exact = trial % 3 == 0
        u = np.eye(1 << k)[rng.permutation(1 << k)].astype(complex) if exact else W.random_unitary(k, rng)
        psi = W.random_state(n, rng).astype(np.complex64)
        s = svlib.StateVector(n, "c64").load(psi)
        s.apply_gate(u, tuple(q[:k]), tuple(q[k:]))
        got, want = s.numpy(), reference(psi.astype(np.complex128), n, u, q[:k], q[k:])
        if exact:
            assert np.array_equal(got, want.astype(np.complex64))
        # 2^k products summed one by one
        assert np.max(np.abs(got - want)) <= (2 << k) * np.finfo(np.float32).eps * np.max(np.abs(psi))
        s.close()
