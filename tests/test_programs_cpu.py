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
    L.program_area.restype = L.reduction_area.restype = C.c_uint64
    L.plan_fmas.restype = C.c_double
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


@pytest.mark.parametrize("dt", [SV_C64, SV_C128])
def test_moved_gates_are_no_arithmetic(tool, dt):
    """A permutation run adds no multiply-adds to the dense gates around it."""
    from paper_2106_13995_gb300 import sim
    n = 24
    rng = np.random.default_rng(3)
    head, run = dense(n, 6, 3, rng), toffolis(n, 300, rng)
    _, flags = build(tool, W.Circuit(n, head + run), dt)
    assert any(f & MOVES for f in flags)
    count = [tool.plan_fmas(C.byref(sim.marshal(W.Circuit(n, ops)).c), dt) for ops in (head, head + run, run)]
    assert count[0] == count[1] > 0 and count[2] == 0


# ---- gradients ----------------------------------------------------------------
def ansatz(n, layers, entangle, fixed=()):
    """RY and RZ on every qubit behind `fixed` gates, then two-qubit gates."""
    ops, np_ = [], 0
    for k in range(layers):
        for q in range(n):
            ops += [W.Op(f, (q,)) for f in fixed]
            for r in ("RY", "RZ"):
                ops.append(W.Op(r, (q,), param=np_))
                np_ += 1
        ops += entangle(k)
    return W.Circuit(n, ops, n_params=np_)


def gradient(tool, c, sets, dt=SV_C64):
    """(passes a gradient launches, whether they are made of sites); it must
    fit the workspace."""
    from paper_2106_13995_gb300 import _native as N, sim
    m, p, t = sim.marshal(c), np.ones(max(1, c.n_params)), W.tfim(c.n_qubits)
    terms, sites = (N.SvPauliTerm * len(t))(*[N.SvPauliTerm(*x) for x in t]), C.c_int()
    prog, acc = C.c_uint64(), C.c_uint64()
    n = tool.gradient_passes(C.byref(m.c), p.ctypes.data_as(C.c_void_p), terms, len(t), sets, dt, C.byref(sites),
                             C.byref(prog), C.byref(acc))
    assert n > 0, n
    assert prog.value <= tool.program_area() and acc.value <= tool.reduction_area(c.n_qubits)
    return n, bool(sites.value)


@pytest.mark.parametrize("n,sets,layers", [(16, 1, 6), (20, 64, 10), (26, 1, 6)])
def test_fixed_gates_do_not_cut_gradients_into_many_passes(tool, n, sets, layers):
    """Sites are kept where what they fold is worth the launches they add to a
    plan of single gates."""
    def ladder(gate):
        return lambda k: [W.Op(gate, (q, q + 1)) if gate != "X" else W.Op("X", (q + 1,), (q,)) for q in range(n - 1)]

    def bricks(k):
        return [W.Op("CZ", (q, q + 1)) for q in range(k % 2, n - 1, 2)]

    plain = gradient(tool, ansatz(n, layers, ladder("CZ")), sets)
    brick = gradient(tool, ansatz(n, layers, bricks), sets)
    assert not plain[1] and not brick[1] and brick[0] <= plain[0] <= 40
    cnots, sites = gradient(tool, ansatz(n, layers, ladder("X")), sets)
    assert sites and cnots <= 1.25 * plain[0]
    mixed, sites = gradient(tool, ansatz(n, layers, ladder("X"), ("H",)), sets)
    assert 16 * (mixed - plain[0]) <= 4 * 2 * n * layers + 3 * (n - 1) * layers or not sites


@pytest.mark.parametrize("dt", [SV_C64, SV_C128])
def test_deep_gradients_fit_as_single_gates(tool, dt):
    """RX and a Toffoli in turn on three qubits: an op of 128 bytes a sweep and
    two matrices of 32 for each pair in sites, 256 bytes in all as single gates
    (384 in complex128)."""
    depth = 30000 if dt == SV_C64 else 20000
    ops = []
    for k in range(depth):
        a, b, d = k % 3, (k + 1) % 3, (k + 2) % 3
        ops += [W.Op("RX", (a,), param=k), W.Op("X", (b,), (a, d))]
    c = W.Circuit(6, ops, n_params=depth)
    gradient(tool, c, 1, dt)


@pytest.mark.parametrize("dt", [SV_C64, SV_C128])
def test_accumulators_leave_room_for_every_parameter(tool, dt):
    """As many parameters as the reduction area holds beside the energy, most of
    them without a gate."""
    n, sets = 8, 64
    c = W.Circuit(n, [W.Op("RX", (q,), param=q) for q in range(n)],
                  n_params=tool.reduction_area(n) // 8 // sets - 1)
    gradient(tool, c, sets, dt)
