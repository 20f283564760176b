"""Exact tensor-core passes of complex128 states against the FP64 oracle."""
import numpy as np
import pytest

import workloads as W
from conftest import fidelity_metrics

pytestmark = pytest.mark.gpu


def check(oracle, want, got, gates):
    """A block rounds each amplitude once relative to its group (2^-53, plus
    2^-56 of the group's norm), and the oracle a few times per gate: random
    walks of at most 8 sqrt(gates) units of the largest amplitude."""
    _, amp = fidelity_metrics(want, got)
    assert amp <= 8 * np.sqrt(gates) * 2.0 ** -53 * np.max(np.abs(want)), amp


@pytest.mark.parametrize("n", [13, 14, 15, 17, 20, 21])
def test_dense_blocks(svlib, oracle, n):
    """Haar-random 5-qubit blocks on every kind of target set (low, high,
    spread), and smaller ones that are padded: more than one pass, and at 20
    and 21 qubits more than one tile per SM."""
    rng = np.random.default_rng(n)
    c = W.Circuit(n)
    sets = [(0, 1, 2, 3, 4), tuple(range(n - 5, n)), (0, n - 1, 3, 8, 6)]
    sets += [tuple(int(q) for q in rng.choice(n, size=int(rng.integers(1, 6)), replace=False)) for _ in range(25)]
    for t in sets:
        c.ops.append(W.Op("MATRIX", t, matrix=W.random_unitary(len(t), rng)))
    psi0 = W.random_state(n, rng)
    s = svlib.StateVector(n, "c128").load(psi0)
    s.apply_circuit(c)
    check(oracle, oracle.run(c, psi0), s.numpy(), len(sets))
    assert abs(s.norm2() - 1) <= 1e-14
    s.close()


@pytest.mark.parametrize("n", [14, 16, 19])
def test_circuits(svlib, oracle, n):
    for c in (W.random_u3_cz(n, 12, n), W.qft(n), W.remove_qubits(W.grid_random(5, 6, 12, 1), 30 - n, 5)):
        s = svlib.StateVector(n, "c128").set_basis(3)
        psi0 = np.zeros(1 << n, dtype=complex)
        psi0[3] = 1
        check(oracle, oracle.run(c, psi0), s.apply_circuit(c).numpy(), len(c.ops))
        s.close()


def test_states_of_every_scale(svlib, oracle):
    """One amplitude, amplitudes over 80 binades, a scaled state, zeros, and
    NaN: what a group without it holds is unchanged by it."""
    n = 14
    rng = np.random.default_rng(2)
    c = W.Circuit(n)
    for _ in range(6):
        t = tuple(int(q) for q in rng.choice(n, size=5, replace=False))
        c.ops.append(W.Op("MATRIX", t, matrix=W.random_unitary(5, rng)))
    z = W.random_state(n, rng)
    one = np.zeros(1 << n, dtype=complex)
    one[4097] = 1j
    for psi0 in (one, z * 2.0 ** rng.integers(-80, 1, 1 << n), z * 2.0 ** -600, z * 2.0 ** 900):
        s = svlib.StateVector(n, "c128").load(psi0)
        check(oracle, oracle.run(c, psi0 / np.max(np.abs(psi0))), s.apply_circuit(c).numpy() / np.max(np.abs(psi0)), 6)
        s.close()
    s = svlib.StateVector(n, "c128").load(np.zeros(1 << n))
    assert not np.any(s.apply_circuit(c).numpy())
    one_block = W.Circuit(n, [W.Op("MATRIX", (0, 1, 2, 3, 13), matrix=W.random_unitary(5, rng))])
    bad = z.copy()
    bad[5] = np.nan
    got = s.load(bad).apply_circuit(one_block).numpy()
    group = np.array([y | (h << 13) for h in (0, 1) for y in range(16)])
    rest = np.setdiff1d(np.arange(1 << n), group)
    want = oracle.run(one_block, z)
    assert np.all(np.isnan(got[group])) and np.max(np.abs(got[rest] - want[rest])) <= 1e-15
    s.close()


def test_runs_are_the_same_and_batches_too(svlib):
    """The same bits on every call, with another state's program in between,
    and in a batched call recorded as a graph."""
    import ctypes as C
    from paper_2106_13995_gb300 import _native as N
    c, d = W.random_u3_cz(14, 8, 1), W.random_u3_cz(14, 8, 2)
    s = svlib.StateVector(14, "c128")
    a = s.set_basis(0).apply_circuit(c).numpy()
    s.set_basis(0).apply_circuit(d)
    assert np.array_equal(s.set_basis(0).apply_circuit(c).numpy(), a)
    ss = [svlib.StateVector(14, "c128").set_basis(0) for _ in range(2)]
    ms = [svlib.marshal(x) for x in (c, d)]
    hs = (C.c_void_p * 2)(*[x.h.value for x in ss])
    cs = (C.POINTER(N.SvCircuit) * 2)(*[C.pointer(m.c) for m in ms])
    o = svlib.options(mode=N.SV_MODE_TILED_GRAPH)
    N.check(N.lib().sv_apply_circuit_batch(hs, 2, cs, None, C.byref(o)))
    ss[0].synchronize()
    assert np.array_equal(ss[0].numpy(), a)


def test_long_programs_keep_the_cuda_cores(svlib, oracle):
    """More blocks than the program area holds operands for (56 KB each)."""
    n = 14
    rng = np.random.default_rng(8)
    c = W.Circuit(n)
    for i in range(160):
        t = tuple(int(q) for q in rng.choice(n, size=5, replace=False))
        c.ops.append(W.Op("MATRIX", t, matrix=W.random_unitary(5, rng)))
    s = svlib.StateVector(n, "c128").set_basis(0)
    check(oracle, oracle.run(c), s.apply_circuit(c).numpy(), 16 * len(c.ops))
    s.close()
