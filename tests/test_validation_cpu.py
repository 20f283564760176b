"""Malformed circuits are refused before their arrays are read."""
import os
import subprocess
import sys

import pytest

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
