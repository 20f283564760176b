"""Exact tensor-core passes of complex128 states on circuits that qualify for
them: target sets, tiles per SM, scales, and batches recorded as a graph."""
import ctypes as C

import numpy as np
import pytest

import oz_cases
import workloads as W

pytestmark = pytest.mark.gpu


def mixing(n, sets, seed):
    """Per set of up to 5 qubits: H and SX on all of them around random phases
    and CZ, entries of one magnitude."""
    rng = np.random.default_rng(seed)
    c = W.Circuit(n)
    for t in sets:
        c.ops += [W.Op("H", (q,)) for q in t]
        c.ops += [W.Op("RZ", (q,), angles=(float(rng.uniform(0, 6)),)) for q in t]
        c.ops += [W.Op("CZ", (a, b)) for a, b in zip(t, t[1:])]
        c.ops += [W.Op("SX", (q,)) for q in t]
    return c


def target_sets(n, count, seed):
    rng = np.random.default_rng(seed)
    sets = [(0, 1, 2, 3, 4), tuple(range(n - 5, n)), (0, n - 1, 3, 8, 6)]
    return sets + [tuple(int(q) for q in rng.choice(n, size=int(rng.integers(2, 6)), replace=False)) for _ in range(count)]


def tensor(s, c):
    """Whether every block is planned as one of 5 qubits on the tensor cores."""
    return s.plan_fmas(c) == 128.0 * s.plan_info(c)[0]


@pytest.mark.parametrize("n", [14, 15, 17, 20, 21])
def test_target_sets(svlib, oracle, n):
    c = mixing(n, target_sets(n, 22, n), n)
    psi0 = W.random_state(n, np.random.default_rng(n)) * 2.0 ** np.random.default_rng(1).integers(-40, 1, 1 << n)
    s = svlib.StateVector(n, "c128")
    assert tensor(s, c)
    oz_cases.check(oracle, c, psi0, s.load(psi0).apply_circuit(c).numpy(), n)
    s.close()


@pytest.mark.parametrize("n", [18, 22])
def test_grid_circuits(svlib, oracle, n):
    c = W.remove_qubits(W.grid_random(5, 6, 10, 3), 30 - n, 7)
    s = svlib.StateVector(n, "c128")
    assert tensor(s, c)
    psi0 = np.zeros(1 << n, dtype=complex)
    psi0[3] = 1
    oz_cases.check(oracle, c, psi0, s.set_basis(3).apply_circuit(c).numpy(), n)
    s.close()


@pytest.mark.parametrize("scale", [2.0 ** -600, 2.0 ** 900, 0.0])
def test_scales(svlib, oracle, scale):
    n = 14
    c = mixing(n, target_sets(n, 6, 2), 2)
    psi0 = W.random_state(n, np.random.default_rng(5))
    s = svlib.StateVector(n, "c128")
    assert tensor(s, c)
    got = s.load(psi0 * scale).apply_circuit(c).numpy()
    if scale == 0:
        assert not np.any(got)
    else:
        assert np.array_equal(got / scale, s.load(psi0).apply_circuit(c).numpy())   # powers of two
    s.close()


def test_batches_as_launches_and_as_a_graph(svlib):
    """A layout's first call goes as launches, its second records a graph, its
    third replays it: the same bits as single circuits each time."""
    from paper_2106_13995_gb300 import _native as N
    cs = [mixing(n, target_sets(n, 8, n), n) for n in (14, 16, 15)]
    ms, want = [svlib.marshal(c) for c in cs], []
    for c in cs:
        s = svlib.StateVector(c.n_qubits, "c128").set_basis(0)
        assert tensor(s, c)
        want.append(s.apply_circuit(c).numpy())
        s.close()
    ss = [svlib.StateVector(c.n_qubits, "c128") for c in cs]
    hs = (C.c_void_p * len(ss))(*[s.h.value for s in ss])
    ptrs = (C.POINTER(N.SvCircuit) * len(ss))(*[C.pointer(m.c) for m in ms])
    o = svlib.options(mode=N.SV_MODE_TILED_GRAPH)
    for call in range(3):
        for s in ss:
            s.set_basis(0)
        N.check(N.lib().sv_apply_circuit_batch(hs, len(ss), ptrs, None, C.byref(o)))
        ss[0].synchronize()
        for s, w in zip(ss, want):
            assert np.array_equal(s.numpy(), w), call
