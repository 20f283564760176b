"""The exact tensor-core blocks' arithmetic without a GPU: digits, kept digit
products and join (oz_digits.cuh, and the packed operand in its core-matrix
layout) against extended precision."""
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
    lib, src = os.path.join(out, "libozemu.so"), os.path.join(HERE, "host", "oz_emulator.cu")
    if not os.path.exists(lib) or any(os.path.getmtime(d) > os.path.getmtime(lib) for d in [src] + objs):
        subprocess.check_call([b.nvcc(), *b.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                               "-I", os.path.join(ROOT, "include"), "-o", lib, src, *objs])
    L = C.CDLL(lib)
    L.oz_block.argtypes = [C.c_void_p] * 4
    return L


def block(emu, u, x):
    u = np.ascontiguousarray(u, dtype=np.complex128)
    x = np.ascontiguousarray(x, dtype=np.complex128)
    out, worst = np.zeros(32, dtype=np.complex128), np.zeros(2)
    rc = emu.oz_block(u.ctypes.data, x.ctypes.data, out.ctypes.data, worst.ctypes.data)
    return rc, out, worst


def states(rng):
    """Dense, spread over 40 binades, one entry, denormals, largest finite."""
    z = rng.standard_normal(32) + 1j * rng.standard_normal(32)
    yield z
    yield z * 2.0 ** rng.integers(-40, 1, 32)
    e = np.zeros(32, dtype=complex)
    e[int(rng.integers(32))] = 2.0 ** -0.5
    yield e
    yield np.full(32, (1 + 1j) * (1 - 2.0 ** -50))    # every number near a power of two
    yield z * 2.0 ** -1060
    yield z * 2.0 ** 1018
    yield np.zeros(32, dtype=complex)


@pytest.mark.parametrize("seed", range(8))
def test_error_is_one_rounding(emu, seed):
    """Digits keep 62 bits of the largest number of a row and of the matrix,
    the dropped weights lie 2^-58 below, and the result is rounded once: at
    most 2^-53 of a result (itself at most the row's norm) plus 2^-56 of the
    norm.  Sums of weight at most 4 stay within FP32's exact integers."""
    rng = np.random.default_rng(seed)
    a, b = W.random_unitary(2, rng), W.random_unitary(3, rng)
    h = np.array([[1, 1], [1, -1]]) / np.sqrt(2)
    h5 = h
    for _ in range(4):
        h5 = np.kron(h5, h)
    qft = np.exp(2j * np.pi * np.outer(np.arange(32), np.arange(32)) / 32) / np.sqrt(32)
    for u in (W.random_unitary(5, rng), np.kron(a, b), np.kron(np.eye(8), a), h5, qft, np.eye(32)):
        for x in states(rng):
            rc, got, worst = block(emu, u, x)
            assert rc == 0
            assert worst[0] <= 2.0 ** -53 + 2.0 ** -56 or np.max(np.abs(x)) < 2.0 ** -1000
            assert worst[1] <= 2 ** 24
            if np.max(np.abs(x)) < 2.0 ** -1000:   # denormal results: absolute rounding
                assert np.max(np.abs(got - u @ x)) <= 64 * 2.0 ** -1074


def test_exact_cases(emu):
    """Permutations and phases of powers of i move bits; one amplitude times a
    matrix gives that column's entries exactly."""
    rng = np.random.default_rng(1)
    x = rng.standard_normal(32) + 1j * rng.standard_normal(32)
    perm, ph = rng.permutation(32), np.array([1, 1j, -1, -1j])[rng.integers(0, 4, 32)]
    p = np.eye(32)[perm] * ph[perm][:, None]
    rc, got, _ = block(emu, p, x)
    assert rc == 0
    # (the join keeps 2^-58 of the row's largest: numbers within 2^-5 of it keep
    # all 53 bits)
    want = (ph * x)[perm]
    for g, w in ((got.real, want.real), (got.imag, want.imag)):
        big = np.abs(w) >= 2.0 ** -5 * np.max(np.abs(x))
        assert big.sum() > 16 and np.array_equal(g[big], w[big])
    u = W.random_unitary(5, rng)
    e = np.zeros(32)
    e[7] = 1
    rc, got, _ = block(emu, u, e)
    assert rc == 0 and np.max(np.abs(got - u[:, 7])) <= 2.0 ** -61


def test_matrices_that_do_not_qualify(emu):
    assert block(emu, np.full((32, 32), np.nan), np.ones(32))[0] == 1
    # every digit of every entry near its largest magnitude
    v = sum(255.0 * 2.0 ** (-9 * i) for i in range(1, 7))
    assert block(emu, np.full((32, 32), v * (1 + 1j)), np.ones(32))[0] == 1
