"""Circuits and states for the accuracy of single amplitudes in complex128:
gates that leave small amplitudes beside large ones unmixed."""
import numpy as np

import workloads as W


def circuits(n, seed):
    """name -> circuit on n qubits."""
    rng = np.random.default_rng(seed)
    q = [int(x) for x in rng.permutation(n)]
    op = W.Op
    out = {"one rotation": [op("RY", (q[0],), angles=(1.1,))],
           "phases": [op("S", (q[0],)), op("T", (q[1],)), op("RZ", (q[2],), angles=(0.7,)), op("CZ", (q[3], q[4]))],
           "controlled": [op("RY", (q[0],), (q[1],), angles=(1.3,)), op("H", (q[2],), (q[3],)),
                          op("PHASE", (q[4],), (q[5],), angles=(0.4,)), op("X", (q[6],), (q[7],))],
           "permutations and one H": [op("H", (q[0],)), op("X", (q[1],), (q[2],)), op("SWAP", (q[3], q[4])),
                                      op("X", (q[5],)), op("FSIM", (q[6], q[7]), angles=(np.pi / 2, np.pi / 6))],
           "small angles": [op("RX", (x,), angles=(float(a),)) for x, a in zip(q, 10.0 ** -np.arange(1, n + 1.0))],
           "matrix with a small entry": [op("MATRIX", (q[0],), matrix=np.array([[1, 1e-9], [-1e-9, 1]], dtype=complex))],
           "unitaries": [op("MATRIX", tuple(q[5 * i:5 * i + 5]), matrix=W.random_unitary(5, rng)) for i in range(2)]}
    out = {k: W.Circuit(n, v) for k, v in out.items()}
    mixed = []
    for _ in range(60):
        t = [int(x) for x in rng.choice(n, size=3, replace=False)]
        mixed.append([op("H", (t[0],)), op("S", (t[0],)), op("SX", (t[0],)), op("X", (t[0],), (t[1],)),
                      op("CZ", (t[0], t[1])), op("RZ", (t[0],), angles=(float(rng.uniform(0, 6)),)),
                      op("FSIM", (t[0], t[1]), angles=(np.pi / 2, np.pi / 6)), op("SWAP", (t[0], t[1])),
                      op("H", (t[0],), (t[1],))][int(rng.integers(9))])
    out["mixed"] = W.Circuit(n, mixed)
    out["grid"] = W.remove_qubits(W.grid_random(5, 6, 6, seed), 30 - n, seed)
    out["qft"] = W.qft(n)
    out["u3 cz"] = W.random_u3_cz(n, 4, seed)
    return out


def states(n, seed):
    """Amplitudes over 80 binades, a large one in every 64, the basis state 0."""
    rng = np.random.default_rng(seed)
    z = W.random_state(n, rng)
    yield z * 2.0 ** rng.integers(-80, 1, 1 << n)
    y = z * 1e-12
    y[::64] = 1
    yield y
    e = np.zeros(1 << n, dtype=complex)
    e[0] = 1
    yield e


def gate_bound(oracle, c, psi0):
    """sum over paths of the magnitudes: what FP64 arithmetic, gate by gate or
    fused, is within rounding of."""
    ops = []
    for o in c.ops:
        u = np.abs(o.matrix if o.name == "MATRIX" else oracle.gate_matrix(o.name, o.angles))
        ops.append(W.Op("MATRIX", o.targets, o.controls, matrix=u.astype(complex)))
    return np.real(oracle.run(W.Circuit(c.n_qubits, ops), np.abs(psi0).astype(complex)))


def check(oracle, c, psi0, got, name):
    """Rounding of a gate stays within 2^-53 of the magnitudes' sum, a block's
    digits within about as much: random walks of 8 units per gate, and the
    oracle's own."""
    want, bound = oracle.run(c, psi0), gate_bound(oracle, c, psi0)
    err = np.abs(got - want)
    tol = 8 * np.sqrt(len(c.ops)) * 2.0 ** -53
    worst = np.max(np.divide(err, bound, out=np.where(err > 0, np.inf, 0), where=bound > 0))
    assert worst <= tol, (name, worst / 2.0 ** -53)
