"""Pauli strings with X and Y factors through the expectation tile passes,
against the FP64 oracle."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def strings(n, rng):
    """Transverse field, XX + YY bonds, masks shared by up to 8 strings (tile
    passes) and by 9 (the table kernel), random strings of weight 1 to 12 (the
    heavier ones span more qubits than a tile), and a diagonal one."""
    t = [(1 << q, 0, 0.5) for q in range(n)]
    for q in range(n - 1):
        b = 3 << q
        t += [(b, 0, 0.3), (b, b, -0.7)]
    for x in (1 << (n - 1), 5, (1 << (n - 1)) | 2):
        t += [(x, int(rng.integers(0, 1 << n)), float(rng.normal())) for _ in range(6)]
    t += [(9, int(rng.integers(0, 1 << n)), float(rng.normal())) for _ in range(9)]
    for w in range(1, min(n, 12) + 1):
        for _ in range(3):
            x = sum(1 << int(q) for q in rng.choice(n, size=w, replace=False))
            t.append((x, int(rng.integers(0, 1 << n)), float(rng.normal())))
    return t + [(0, 3, 0.25)]


@pytest.mark.parametrize("dt,eps", [("c64", 2.0 ** -24), ("c128", 2.0 ** -53)])
@pytest.mark.parametrize("n", [9, 10, 11, 16, 17, 21, 22])
def test_x_and_y_strings(svlib, oracle, dt, eps, n):
    """The widths reach the smallest tile (8 qubits), every tile size up to
    the largest and the table kernel below 10 qubits.  A string's sum over
    pairs is made of products of relative error eps in runs of at most 32
    roundings each, and the runs are added in FP64: at most 64 eps of
    sum |c|."""
    rng = np.random.default_rng(n)
    s = svlib.StateVector(n, dt).load(W.random_state(n, rng))
    psi = s.numpy().astype(np.complex128)
    terms = strings(n, rng)
    scale = sum(abs(c) for _, _, c in terms)
    got, want = s.expect(terms), oracle.expect(psi, terms)
    assert abs(got - want) <= 64 * eps * scale, (got, want)
    # one string at a time, and strings whose value is exactly 1
    for t in terms[:: max(1, len(terms) // 12)]:
        assert abs(s.expect([t]) - oracle.expect(psi, [t])) <= 64 * eps * abs(t[2]), t
    s.set_basis(0).apply_circuit(W.hadamard_all(n))
    assert abs(s.expect([(1 << q, 0, 1.0) for q in range(n)]) - n) <= 4096 * eps * n
    s.close()


def test_many_masks_fold_partial_sums(svlib, oracle):
    """More passes than the workspace holds partial sums for (its 2 MB area):
    strings of weight 6 to 8 rarely share a pass."""
    n = 21
    rng = np.random.default_rng(3)
    s = svlib.StateVector(n, "c64").load(W.random_state(n, rng))
    terms = []
    for _ in range(900):
        x = sum(1 << int(q) for q in rng.choice(n, size=int(rng.integers(6, 9)), replace=False))
        terms.append((x, int(rng.integers(0, 1 << n)), float(rng.normal())))
    want = oracle.expect(s.numpy().astype(np.complex128), terms)
    assert abs(s.expect(terms) - want) <= 64 * 2.0 ** -24 * sum(abs(t[2]) for t in terms)
    s.close()
