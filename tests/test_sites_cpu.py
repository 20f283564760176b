"""The blocks gradient programs are made of, without a GPU: site_blocks of
mixed circuits and of their adjoints, applied by a CPU interpreter
(tests/host/sites_emulator.cu), against the FP64 oracle."""
import ctypes as C
import glob
import os
import subprocess

import numpy as np
import pytest

import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def emu():
    import importlib
    import paper_2106_13995_gb300 as P
    b = importlib.import_module("paper_2106_13995_gb300.buildlib")
    P.build()
    objs = sorted(glob.glob(os.path.join(b.OUT_DIR, "*.o")))
    out = os.path.join(HERE, "host", "_build")
    os.makedirs(out, exist_ok=True)
    lib, src = os.path.join(out, "libsitesemu.so"), os.path.join(HERE, "host", "sites_emulator.cu")
    if not os.path.exists(lib) or any(os.path.getmtime(d) > os.path.getmtime(lib) for d in [src] + objs):
        subprocess.check_call([b.nvcc(), *b.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                               "-I", os.path.join(ROOT, "include"), "-o", lib, src, *objs])
    L = C.CDLL(lib)
    L.sites_run.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int, C.c_int, C.POINTER(C.c_int)]
    return L


def run(emu, circ, params, psi, reverse, K=2):
    from paper_2106_13995_gb300 import sim
    m = sim.marshal(circ)
    p = np.ascontiguousarray(params, dtype=np.float64)
    out = np.ascontiguousarray(psi, dtype=np.complex128).copy()
    ns = C.c_int()
    nb = emu.sites_run(C.addressof(m.c), p.ctypes.data, out.ctypes.data, int(reverse), K, C.byref(ns))
    assert nb > 0
    return out, nb, ns.value


def mixed(n, count, seed):
    """Parametric rotations, permutations of 1 to 3 and of 4 qubits, named and
    dense gates with and without controls."""
    rng = np.random.default_rng(seed)
    c = W.Circuit(n)
    for _ in range(count):
        r = rng.random()
        q = [int(x) for x in rng.permutation(n)[:5]]
        if r < 0.5:
            c.ops.append(W.Op(("RX", "RY", "RZ", "PHASE")[int(rng.integers(4))], (q[0],), param=c.n_params))
            c.n_params += 1
        elif r < 0.75:
            c.ops.append(W.Op("X", (q[0],), tuple(q[1:1 + int(rng.integers(0, 4))])))
        elif r < 0.8:
            c.ops.append(W.Op("SWAP", tuple(q[:2])))
        elif r < 0.9:
            c.ops.append(W.Op("U3", (q[0],), tuple(q[1:1 + int(rng.integers(0, 3))]),
                              tuple(float(a) for a in rng.uniform(-3, 3, 3))))
        else:
            k = int(rng.integers(2, 4))
            c.ops.append(W.Op("MATRIX", tuple(q[:k]), matrix=W.random_unitary(k, rng)))
    return c


@pytest.mark.parametrize("seed", range(12))
def test_mixed_circuits_both_ways(emu, oracle, seed):
    n = 5 + seed % 4
    c = mixed(n, 90, seed)
    rng = np.random.default_rng(seed)
    p, psi0 = rng.uniform(-3, 3, max(1, c.n_params)), W.random_state(n, rng)
    want = oracle.run(c, psi0, params=p)
    for K in (1, 2, 3):
        got, _, _ = run(emu, c, p, psi0, False, K)
        assert np.max(np.abs(got - want)) <= 1e-13
        back, _, _ = run(emu, c, p, want, True, K)
        assert np.max(np.abs(back - psi0)) <= 1e-13


def test_ansatz_takes_one_op_per_two_qubits_and_layer(emu, oracle):
    """RY, RZ on every qubit, then a CNOT ladder: one site per qubit and layer,
    about n / 2 ops a layer in both directions."""
    n, layers = 10, 4
    c = W.hea(n, layers)
    p = W.hea_params(1, c.n_params, 1)[0]
    psi0 = W.random_state(n, np.random.default_rng(1))
    for reverse in (False, True):
        _, nb, ns = run(emu, c, p, psi0, reverse)
        assert ns == n * layers
        assert nb <= (n // 2 + 1) * layers + 1
