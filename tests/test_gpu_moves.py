"""Permutation runs as moves against the table passes of the same gates (a
fusion width asked for keeps those): moved amplitudes are equal bit for bit."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def reversible(B, n, count, rng):
    """X, CNOT, Toffoli, SWAP, controlled SWAP and 3-qubit permutations, most of
    them moving n - 4 of the qubits (so that a run is a few passes)."""
    c = B.Circuit(n)
    some = np.concatenate([np.arange(5), 5 + rng.permutation(n - 5)[:n - 9]])
    for i in range(count):
        of = np.arange(n) if i % 50 == 49 else some
        t = [int(x) for x in rng.permutation(of)[:3]]
        q = t + [int(x) for x in rng.permutation(n) if x not in t][:5]
        kind = int(rng.integers(0, 6))
        if kind == 0:
            c.append("X", (q[0],), (), ())
        elif kind <= 2:
            c.append("X", (q[0],), (), tuple(q[3:3 + kind]))
        elif kind == 3:
            c.append("X", (q[0],), (), tuple(q[3:3 + int(rng.integers(3, 6))]))
        elif kind == 4:
            c.append("SWAP", tuple(q[:2]), (), tuple(q[3:3 + int(rng.integers(0, 2))]))
        else:
            c.unitary(np.eye(8, dtype=complex)[rng.permutation(8)], *q[:3])
    return c


def dense(svlib, n, dt, seed):
    s = svlib.StateVector(n, dt)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s.amps.normal_(generator=g)
    return s


def both(svlib, n, dt, m, seed):
    a, b = dense(svlib, n, dt, seed), dense(svlib, n, dt, seed)
    a.apply_circuit(m)
    b.apply_circuit(m, opts=svlib.options(fusion_k=3))
    torch.cuda.synchronize()
    eq = torch.equal(a.amps, b.amps)
    plans = a.plan_info(m)[1], b.plan_info(m, opts=svlib.options(fusion_k=3))[1]
    a.close()
    b.close()
    return eq, plans


@pytest.mark.parametrize("n,dt", [(14, "c64"), (15, "c64"), (17, "c64"), (22, "c64"), (25, "c64"), (26, "c64"),
                                  (15, "c128"), (21, "c128"), (24, "c128"), (25, "c128")])
def test_runs_equal_table_passes(svlib, n, dt):
    """From no scratch (14 qubits) over the smallest chunks to the largest, several
    passes each."""
    from paper_2106_13995_gb300 import circuit as B
    rng = np.random.default_rng(n)
    m = svlib.marshal(reversible(B, n, 200, rng))
    eq, (moves, tables) = both(svlib, n, dt, m, n)
    assert eq
    assert moves < tables or n < 15


def test_dense_gates_around_a_run(svlib):
    """Hadamards, a run, rotations, a run: the parts in order (the dense parts
    are the same passes on both routes up to the fusion across their borders)."""
    from paper_2106_13995_gb300 import circuit as B
    n = 18
    for dt, tol in (("c64", 2e-6), ("c128", 1e-14)):
        rng = np.random.default_rng(3)
        c = B.Circuit(n)
        for part in range(2):
            for q in range(n):
                c.append("H" if part == 0 else "RY", (q,), () if part == 0 else (0.1 * q + 0.2,), ())
            for op in reversible(B, n, 150, rng).ops:
                c.ops.append(op)
        m = svlib.marshal(c)
        a, b = (svlib.StateVector(n, dt).set_basis(5) for _ in range(2))
        a.apply_circuit(m)
        b.apply_circuit(m, opts=svlib.options(fusion_k=3))
        assert a.plan_info(m)[1] < b.plan_info(m, opts=svlib.options(fusion_k=3))[1]
        d = float((a.amps - b.amps).norm() / b.amps.norm())
        assert d < tol


def test_in_batches_graphs_and_small_workspaces(svlib):
    """Runs in a batch of states (each with its own scratch), replayed from a
    graph, and a state whose workspace has no room for the scratch."""
    from paper_2106_13995_gb300 import _native as N
    from paper_2106_13995_gb300 import circuit as B
    rng = np.random.default_rng(9)
    ns = [14, 16, 12, 18, 23]
    ms = [svlib.marshal(reversible(B, n, 100, rng)) for n in ns]
    o = svlib.options(mode=N.SV_MODE_TILED_GRAPH)
    a = [dense(svlib, n, "c64", n) for n in ns]
    b = [dense(svlib, n, "c64", n) for n in ns]
    hs = (C.c_void_p * len(a))(*[s.h.value for s in a])
    cs = (C.POINTER(N.SvCircuit) * len(ms))(*[C.pointer(m.c) for m in ms])
    for _ in range(3):
        N.check(N.lib().sv_apply_circuit_batch(hs, len(a), cs, None, C.byref(o)))
        for s, m in zip(b, ms):
            s.apply_circuit(m, opts=svlib.options(fusion_k=3))
    for s, t in zip(a, b):
        assert torch.equal(s.amps, t.amps)
    # the smallest workspace that sv_create takes
    n, m = 18, ms[3]
    amps = a[3].amps.clone()
    lo, hi = 1, N.lib().sv_workspace_bytes(n, N.SV_C64)
    ws = torch.empty(hi, dtype=torch.uint8, device="cuda")
    h = C.c_void_p()

    def create(size):
        return N.lib().sv_create(n, N.SV_C64, amps.data_ptr(), amps.numel() * 4, ws.data_ptr(), size,
                                 C.c_void_p(torch.cuda.current_stream().cuda_stream), C.byref(h))
    while lo < hi:
        mid = (lo + hi) // 2
        if create(mid) == N.SV_OK:
            N.lib().sv_destroy(h)
            hi = mid
        else:
            lo = mid + 1
    assert create(lo) == N.SV_OK and lo < N.lib().sv_workspace_bytes(n, N.SV_C64)
    N.check(N.lib().sv_apply_circuit(h, m.ref(), None, None))
    a[3].apply_circuit(m)
    torch.cuda.synchronize()
    assert torch.equal(amps, a[3].amps)
    N.lib().sv_destroy(h)


@pytest.mark.parametrize("n,dt", [(15, "c64"), (16, "c128"), (19, "c64")])
def test_product_states_before_a_run(svlib, oracle, n, dt):
    """Single-qubit gates on a known basis state (with a phase of its own), then
    a run: against the same circuit on a state the handle does not know, and the
    oracle's product; the state is not taken for known afterwards."""
    from paper_2106_13995_gb300 import _native as N
    from paper_2106_13995_gb300 import circuit as B
    rng = np.random.default_rng(n)
    c = B.Circuit(n)
    for q in range(n):
        for name in ("H", "U3", "T", "X")[:int(rng.integers(0, 5))]:
            c.append(name, (q,), tuple(rng.uniform(0, 6, 3)) if name == "U3" else (), ())
    for op in reversible(B, n, 150, rng).ops:
        c.ops.append(op)
    ph = B.Circuit(n).append("S", (1,), (), ())
    m, p = svlib.marshal(c), svlib.marshal(ph)
    index = int(rng.integers(1 << n)) | 2
    a, b = (svlib.StateVector(n, dt).set_basis(index) for _ in range(2))
    for s in (a, b):
        s.apply_circuit(p)
    N.check(N.lib().sv_mark_modified(b.h))
    for s in (a, b):
        s.apply_circuit(m)
    want = b.numpy().astype(np.complex128)
    # a product of n factors rounded twice against tile passes of 3-qubit blocks
    tol = 64 * np.finfo(np.float32 if dt == "c64" else np.float64).eps
    assert np.max(np.abs(a.numpy() - want)) <= tol * np.max(np.abs(want))
    for s in (a, b):
        s.apply_circuit(m)
    want = b.numpy().astype(np.complex128)
    assert np.max(np.abs(a.numpy() - want)) <= 4 * tol * np.max(np.abs(want))


@pytest.mark.parametrize("n,dt", [(16, "c64"), (16, "c128")])
def test_recorded_launches_replay_on_other_states(svlib, n, dt):
    """Dense gates, a run and dense gates again, recorded by the caller from a
    known basis state: replays act on whatever the state holds (no product state
    is recorded), as the same calls do."""
    from paper_2106_13995_gb300 import circuit as B
    rng = np.random.default_rng(n)
    c = B.Circuit(n)
    for q in range(n):
        c.append("H", (q,), (), ())
    for op in reversible(B, n, 150, rng).ops:
        c.ops.append(op)
    for q in range(n):
        c.append("RY", (q,), (0.1 + 0.2 * q,), ())
    m = svlib.marshal(c)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        s = svlib.StateVector(n, dt, stream=side)
        s.set_basis(3)
        s.amps.zero_()
        s.amps[6] = 1.0
        s.apply_circuit(m, opts=svlib.options())
        from paper_2106_13995_gb300 import _native as N
        N.check(N.lib().sv_mark_modified(s.h))
        s.apply_circuit(m)          # the program that is recorded, resident
        s.set_basis(3)
        side.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            s.apply_circuit(m)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(1)
        s.amps.normal_(generator=gen)
        t = svlib.StateVector(n, dt, stream=side)
        t.amps.copy_(s.amps)
        g.replay()
        t.apply_circuit(m)
        side.synchronize()
        assert torch.equal(s.amps, t.amps)
