"""Which tiles small states take: permutation runs and wide blocks the large
ones where these take fewer passes or fill them."""
import numpy as np
import pytest

import workloads as W
from test_programs_cpu import SV_C64, SV_C128, build, toffolis, tool  # noqa: F401

OZ, MOVES = 0x1000, 0x2000   # kPassOz, kPassMoves


def large(dt):
    from paper_2106_13995_gb300 import sim
    return sim.options(fusion_k=3, tile_m=13 if dt == SV_C64 else 12)


@pytest.mark.parametrize("n", [8, 11, 12, 13, 14, 16, 17])
@pytest.mark.parametrize("dt", [SV_C64, SV_C128])
def test_permutation_circuits(tool, dt, n):  # noqa: F811
    """300 Toffolis: no more passes than in large tiles, none of them moves
    (33 us each against 8)."""
    c = W.Circuit(n, toffolis(n, 300, np.random.default_rng(n)))
    want, got = build(tool, c, dt, large(dt))[1], build(tool, c, dt)[1]
    assert len(got) == len(want) and not any(f & MOVES for f in got)


@pytest.mark.parametrize("n", [13, 14, 16])
@pytest.mark.parametrize("dt", [SV_C64, SV_C128])
def test_runs_between_dense_gates(tool, dt, n):  # noqa: F811
    """The gates around a long run keep their small tiles, the run takes large
    ones."""
    h, run = W.hadamard_all(n).ops, toffolis(n, 300, np.random.default_rng(n))
    alone = build(tool, W.Circuit(n, run), dt, large(dt))[1]
    around = build(tool, W.Circuit(n, h), dt)[1]
    got = build(tool, W.Circuit(n, h + run + h), dt)[1]
    assert len(got) == len(alone) + 2 * len(around)


@pytest.mark.parametrize("dt", [SV_C64, SV_C128])
def test_short_runs_stay_with_the_gates_around_them(tool, dt):  # noqa: F811
    """Layers of rotations and CNOT ladders: as without a rule for runs."""
    n, ops = 16, []
    rng = np.random.default_rng(1)
    for _ in range(6):
        ops += [W.Op("RY", (q,), angles=(float(a),)) for q, a in enumerate(rng.uniform(0.01, 0.02, n))]
        ops += [W.Op("X", (q + 1,), (q,)) for q in range(n - 1)]
    from paper_2106_13995_gb300 import sim
    small = sim.options(fusion_k=3, tile_m=11) if dt == SV_C64 else sim.options(fusion_k=2, tile_m=7)
    assert len(build(tool, W.Circuit(n, ops), dt)[1]) == len(build(tool, W.Circuit(n, ops), dt, small)[1])


@pytest.mark.parametrize("n", [17, 18, 20])
def test_wide_blocks(tool, n):  # noqa: F811
    """Dense 5-qubit blocks that do not qualify for the tensor cores."""
    c = W.block_chain(n, 20, 0)
    assert len(build(tool, c, SV_C128)[1]) == len(build(tool, c, SV_C128, large(SV_C128))[1])


@pytest.mark.parametrize("n", [14, 17, 20, 22, 24])
def test_moves_with_few_dense_gates_keep_fp64(tool, n):  # noqa: F811
    """A GHZ state: one Hadamard and permutations.  With as much dense work as
    moves the tensor cores stay."""
    assert not any(f & OZ for f in build(tool, W.ghz(n), SV_C128)[1])
    c = W.concat(W.ghz(n), W.remove_qubits(W.grid_random(5, 6, 12, 1), 30 - n, 3))
    assert all(f & OZ for f in build(tool, c, SV_C128)[1])


def test_three_qubits_are_one_block(tool):  # noqa: F811
    """A complex128 circuit of 3 qubits: no more ops than with fused triples."""
    c = W.random_u3_cz(3, 40, 1)
    assert build(tool, c, SV_C128)[0] <= build(tool, c, SV_C128, large(SV_C128))[0]
