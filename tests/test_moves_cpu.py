"""Permutation runs without a GPU: gates as multi-controlled X, cut into passes,
every pass's descriptor followed as the kernel follows it."""
import ctypes as C
import glob
import os
import subprocess

import numpy as np
import pytest

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
    lib, src = os.path.join(out, "libmovesemu.so"), os.path.join(HERE, "host", "moves_emulator.cu")
    if not os.path.exists(lib) or any(os.path.getmtime(d) > os.path.getmtime(lib) for d in [src] + objs):
        subprocess.check_call([b.nvcc(), *b.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                               "-I", os.path.join(ROOT, "include"), "-o", lib, src, *objs])
    L = C.CDLL(lib)
    L.moves_emulate.argtypes = [C.c_int] * 3 + [C.c_void_p] * 5
    return L


@pytest.mark.parametrize("n,m,ngates,seed", [(12, 12, 60, 0), (14, 14, 80, 1), (14, 12, 40, 2), (16, 13, 120, 3),
                                             (15, 12, 300, 4), (13, 12, 12, 5)])
def test_moves_follow_the_gates(emu, n, m, ngates, seed):
    """Random permutations of 1 to 3 qubits with up to 8 controls: the source
    index of every amplitude, against the gates applied one by one."""
    rng = np.random.default_rng(seed)
    ks, ncs, qs, perms = [], [], [], []
    idx = np.arange(1 << n)   # idx[y]: where the amplitude at y goes
    for _ in range(ngates):
        k, nc = int(rng.integers(1, 4)), int(rng.integers(0, 4) if rng.random() < 0.9 else rng.integers(4, 9))
        q = rng.permutation(n)[:k + nc]
        p = rng.permutation(1 << k) if rng.random() < 0.5 else np.arange(1 << k) ^ ((1 << k) - 1)
        ks.append(k)
        ncs.append(nc)
        qs.extend(int(x) for x in q)
        perms.extend([int(x) for x in p] + [0] * (8 - (1 << k)))
        c = np.zeros_like(idx)
        for j in range(k):
            c |= ((idx >> q[j]) & 1) << j
        on = np.ones(idx.shape, dtype=bool)
        for j in range(k, k + nc):
            on &= ((idx >> q[j]) & 1) == 1
        r, new = p[c], idx.copy()
        for j in range(k):
            new = (new & ~(1 << int(q[j]))) | (((r >> j) & 1) << int(q[j]))
        idx = np.where(on, new, idx)
    want = np.empty_like(idx)
    want[idx] = np.arange(1 << n)
    a = [np.array(x, dtype=np.int32) for x in (ks, ncs, qs, perms)]
    src = np.zeros(1 << n, dtype=np.uint32)
    rc = emu.moves_emulate(n, m, ngates, *[x.ctypes.data for x in a], src.ctypes.data)
    assert rc >= 1 and np.array_equal(src, want)
