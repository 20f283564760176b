"""Batched calls over many small states: more passes than the first state's
workspace holds tables for, and the lines between queue and launches."""
import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TABLE_AREA, DESCRIPTOR = 2 << 20, 200   # bytes: the reduction area of small states, one pass's entry


def batch(svlib, N, ss, ms, mode):
    h = (C.c_void_p * len(ss))(*[s.h.value for s in ss])
    cs = (C.POINTER(N.SvCircuit) * len(ms))(*[C.pointer(m.c) for m in ms])
    N.check(N.lib().sv_apply_circuit_batch(h, len(ss), cs, None, C.byref(svlib.options(mode=mode))))
    N.check(N.lib().sv_synchronize(ss[0].h))


def test_tables_beyond_the_workspace(svlib):
    """The same bits as one call per state, launched, recorded and replayed."""
    from paper_2106_13995_gb300 import _native as N
    n, B = 12, 64
    ss = [svlib.StateVector(n, "c128") for _ in range(B)]
    ms = [svlib.marshal(W.random_u3_cz(n, 150, b % 4)) for b in range(B)]
    assert sum(s.plan_info(m)[1] for s, m in zip(ss, ms)) * DESCRIPTOR > TABLE_AREA
    psi = [W.random_state(n, np.random.default_rng(b)) for b in range(B)]
    want = [s.load(p).apply_circuit(m).numpy() for s, p, m in zip(ss, psi, ms)]
    for mode in [N.SV_MODE_TILED] + 3 * [N.SV_MODE_TILED_GRAPH]:
        for s, p in zip(ss, psi):
            s.load(p)
        batch(svlib, N, ss, ms, mode)
        for s, w in zip(ss, want):
            assert np.array_equal(s.numpy(), w)
    for s in ss:
        s.close()


@pytest.mark.parametrize("dt,n,B", [("c128", 12, 96), ("c128", 7, 96), ("c64", 14, 41), ("c64", 15, 40), ("c64", 18, 3)])
def test_many_states_as_single_calls(svlib, dt, n, B):
    """Either side of the lines between the queue's CTA sizes and between queue
    and launches: the same bits as one call per state."""
    from paper_2106_13995_gb300 import _native as N
    ss = [svlib.StateVector(n, dt) for _ in range(B)]
    ms = [svlib.marshal(W.random_u3_cz(n, 6, b % 5)) for b in range(B)]
    psi = [W.random_state(n, np.random.default_rng(b)) for b in range(B)]
    want = [s.load(p).apply_circuit(m).numpy() for s, p, m in zip(ss, psi, ms)]
    for mode in [N.SV_MODE_TILED] + 3 * [N.SV_MODE_TILED_GRAPH]:
        for s, p in zip(ss, psi):
            s.load(p)
        batch(svlib, N, ss, ms, mode)
        for s, w in zip(ss, want):
            assert np.array_equal(s.numpy(), w)
    for s in ss:
        s.close()
