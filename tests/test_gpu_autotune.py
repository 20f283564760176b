"""What the autotuner hands back runs the path it found fastest."""
import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["digits", "moves", "tiles"])
def test_the_choice_keeps_the_fastest_path(svlib, what):
    """Exact digits and permutation runs, several times faster than every
    explicit pair, are named by 0 and 0; tile passes by a pair."""
    from paper_2106_13995_gb300 import _native as N
    if what == "digits":
        c, dt = W.remove_qubits(W.grid_random(5, 6, 12, 1), 9, 3), "c128"
    elif what == "moves":
        rng = np.random.default_rng(1)
        q = [rng.choice(25, size=3, replace=False) for _ in range(400)]
        c, dt = W.Circuit(25, [W.Op("X", (int(t[0]),), (int(t[1]), int(t[2]))) for t in q]), "c64"
    else:
        c, dt = W.random_u3_cz(14, 12, 2), "c64"
    s, o = svlib.StateVector(c.n_qubits, dt), svlib.options()
    m = svlib.marshal(c)
    N.check(N.lib().sv_autotune(s.h, m.ref(), C.byref(o)))
    if what == "tiles":
        assert 2 <= o.fusion_k <= 6 and 10 <= o.tile_m <= 14
    else:
        assert (o.fusion_k, o.tile_m) == (0, 0)
    assert s.plan_info(m, opts=o) == s.plan_info(m)
    s.close()
