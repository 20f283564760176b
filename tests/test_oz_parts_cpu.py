"""The accuracy of every amplitude through exact tensor-core programs, without a
GPU: the library's programs interpreted digit by digit."""
import ctypes as C

import numpy as np
import pytest

import oz_cases
from host_tools import load

N = 14


@pytest.fixture(scope="module")
def emu():
    return load("oz_program")


def run(emu, c, psi0):
    from paper_2106_13995_gb300 import sim
    m, psi = sim.marshal(c), np.array(psi0, dtype=np.complex128)
    return emu.oz_program(C.byref(m.c), psi.ctypes.data_as(C.c_void_p)), psi


@pytest.mark.parametrize("name", list(oz_cases.circuits(N, 0)))
def test_small_amplitudes_keep_their_digits(emu, oracle, name):
    c = oz_cases.circuits(N, 0)[name]
    for psi0 in oz_cases.states(N, 1):
        blocks, got = run(emu, c, psi0)
        assert blocks >= 0
        if blocks == 0:
            break   # FP64 arithmetic on the CUDA cores
        oz_cases.check(oracle, c, psi0, got, name)


@pytest.mark.parametrize("name,tensor", [("one rotation", True), ("controlled", True), ("grid", True), ("qft", True),
                                         ("small angles", False), ("matrix with a small entry", False)])
def test_which_circuits_take_the_tensor_cores(emu, name, tensor):
    c = oz_cases.circuits(N, 0)[name]
    blocks, _ = run(emu, c, np.zeros(1 << N))
    assert (blocks > 0) == tensor
