"""Programs as the library builds them, without a GPU: their size against the
workspace's program area."""
import ctypes as C

import numpy as np
import pytest

import workloads as W
from host_tools import load

SV_C64, SV_C128 = 0, 1
OZ, MOVES = 0x1000, 0x2000   # kPassOz, kPassMoves


@pytest.fixture(scope="module")
def tool():
    L = load("program_tool")
    L.program_area.restype = C.c_uint64
    return L


def build(tool, c, dt, opts=None):
    """(bytes of the program area, flags of each pass)"""
    from paper_2106_13995_gb300 import sim
    m = sim.marshal(c)
    end, flags, n = C.c_uint64(), (C.c_uint32 * 4096)(), C.c_int()
    assert tool.program_build(C.byref(m.c), dt, C.byref(opts) if opts else None, C.byref(end), flags, 4096,
                              C.byref(n)) == 0
    return end.value, list(flags[:n.value])


def dense(n, count, k, rng):
    return [W.Op("MATRIX", tuple(int(q) for q in rng.choice(n, size=k, replace=False)), matrix=W.random_unitary(k, rng))
            for _ in range(count)]


def toffolis(n, count, rng):
    qs = [rng.choice(n, size=3, replace=False) for _ in range(count)]
    return [W.Op("X", (int(q[0]),), (int(q[1]), int(q[2]))) for q in qs]


@pytest.mark.parametrize("dt", [SV_C64, SV_C128])
@pytest.mark.parametrize("head", [100, 130, 138, 142, 145])
def test_segments_share_the_program_area(tool, dt, head):
    """A dense stretch, a permutation run, another dense stretch: the first
    one's operands (56 KB a block on the tensor cores) leave room for what
    follows, or the program is built without them."""
    n = 20
    rng = np.random.default_rng(head)
    c = W.Circuit(n, dense(n, head, 5, rng) + toffolis(n, 200, rng) + dense(n, 100, 3, rng))
    end, flags = build(tool, c, dt)
    assert flags and end <= tool.program_area()


def test_a_program_that_fits_keeps_its_paths(tool):
    n = 20
    rng = np.random.default_rng(1)
    c = W.Circuit(n, dense(n, 30, 5, rng) + toffolis(n, 200, rng) + dense(n, 30, 5, rng))
    end, flags = build(tool, c, SV_C128)
    assert end <= tool.program_area() and any(f & MOVES for f in flags)


@pytest.mark.parametrize("dt", [SV_C64, SV_C128])
def test_small_state_plans_take_no_more_than_large_tiles(tool, dt):
    """110000 Toffolis on 12 qubits: one tile holds the state and composes 300
    gates into a table, small default tiles take ops and tables for few each."""
    from paper_2106_13995_gb300 import sim
    n = 12
    c = W.Circuit(n, toffolis(n, 110000, np.random.default_rng(n)))
    large, _ = build(tool, c, dt, sim.options(fusion_k=3, tile_m=13 if dt == SV_C64 else 12))
    small, _ = build(tool, c, dt)
    assert large <= tool.program_area() and small <= tool.program_area()
