"""Malformed circuits are refused before their arrays are read, and circuits on
a known basis state are followed and validated op by op."""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest

import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))

# a matrix pool of one entry whose end is followed by a page nobody may read
RUN = """
import ctypes as C, mmap, sys
sys.path[:0] = [{root!r}, {here!r}]
from host_tools import load
from paper_2106_13995_gb300 import _native as N
tool, libc = load("program_tool"), C.CDLL(None)
libc.mmap.restype = C.c_void_p
libc.mmap.argtypes = [C.c_void_p, C.c_size_t, C.c_int, C.c_int, C.c_int, C.c_long]
page = mmap.PAGESIZE
base = libc.mmap(None, 2 * page, 3, 0x22, -1, 0)
assert libc.mprotect(C.c_void_p(base + page), page, 0) == 0
ops = (N.SvOp * 2)()
ops[0].gate, ops[0].n_targets, ops[0].param = 1, 1, -1
ops[1].gate, ops[1].n_targets, ops[1].param = 0, {targets}, -1
c = N.SvCircuit(n_qubits=9, n_ops=2, n_params=0, ops=ops, matrices=C.cast(base + page - 16, C.POINTER(C.c_double)))
n, end, flags = C.c_int(), C.c_uint64(), (C.c_uint32 * 4)()
sites, prog, acc, term = C.c_int(), C.c_uint64(), C.c_uint64(), (N.SvPauliTerm * 1)(N.SvPauliTerm(0, 1, 1.0))
print(tool.program_build(C.byref(c), 0, None, C.byref(end), flags, 4, C.byref(n)),
      tool.gradient_passes(C.byref(c), None, term, 1, 1, 0, C.byref(sites), C.byref(prog), C.byref(acc)))
"""


@pytest.mark.parametrize("targets", [0, 7, 13, 40, -3])
def test_matrix_sizes_are_checked_before_a_matrix_is_read(targets):
    from host_tools import load
    load("program_tool")   # (built before the other process loads it)
    code = RUN.format(root=os.path.dirname(HERE), here=HERE, targets=targets)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.split() == ["1", "-1"], (r.returncode, r.stdout, r.stderr[-500:])


def random_op(n, rng, n_params):
    """A gate that maps basis states to basis states, of every arity in turn."""
    kind = int(rng.integers(8))
    q = [int(x) for x in rng.permutation(n)]
    if kind == 0:
        return W.Op("X", (q[0],), tuple(q[1:1 + int(rng.integers(4))]))
    if kind == 1:
        return W.Op("RZ", (q[0],), tuple(q[1:1 + int(rng.integers(2))]), param=int(rng.integers(n_params)))
    if kind == 2:
        return W.Op("PHASE", (q[0],), tuple(q[1:1 + int(rng.integers(3))]), angles=(float(rng.uniform(0, 6)),))
    if kind == 3:
        return W.Op("FSIM", (q[0], q[1]), angles=(np.pi / 2, float(rng.uniform(0, 6))))
    if kind == 4:
        return W.Op(["S", "T", "Y", "Z", "SDG"][int(rng.integers(5))], (q[0],), tuple(q[1:1 + int(rng.integers(2))]))
    if kind == 5:
        return W.Op(["SWAP", "CZ"][int(rng.integers(2))], (q[0], q[1]), tuple(q[2:2 + int(rng.integers(2))]))
    k = int(rng.integers(1, 5))   # a monomial matrix
    u = np.zeros((1 << k, 1 << k), dtype=complex)
    u[rng.permutation(1 << k), np.arange(1 << k)] = np.exp(1j * rng.uniform(0, 6, 1 << k))
    return W.Op("MATRIX", tuple(q[:k]), tuple(q[k:k + int(rng.integers(2))]), matrix=u)


@pytest.mark.parametrize("seed", range(6))
def test_basis_states_are_followed_op_by_op(oracle, seed):
    """The index and phase after 80 gates of mixed kinds and arities; a gate
    that spreads the state ends it, a malformed op is refused."""
    from host_tools import load
    from paper_2106_13995_gb300 import sim
    tool, n, rng = load("program_tool"), 8, np.random.default_rng(seed)
    c = W.Circuit(n, [random_op(n, rng, 3) for _ in range(80)], n_params=3)
    p, start = rng.uniform(-3, 3, 3), int(rng.integers(1 << n))
    idx, amp = C.c_uint64(), (C.c_double * 2)()

    def follow(circ):
        m = sim.marshal(circ)
        return tool.follow_basis(C.byref(m.c), p.ctypes.data_as(C.c_void_p), C.c_uint64(start), C.byref(idx), amp)

    assert follow(c) == 1
    psi = np.zeros(1 << n, dtype=complex)
    psi[start] = 1
    want = oracle.run(c, psi, p)
    assert np.count_nonzero(want) == 1 and abs(want[idx.value] - complex(*amp)) <= 1e-13
    assert follow(W.Circuit(n, c.ops + [W.Op("H", (2,))], n_params=3)) == 0
    assert follow(W.Circuit(n, c.ops + [W.Op("RZ", (2,), param=3)], n_params=3)) == -1
