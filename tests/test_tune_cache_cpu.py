"""The autotuner's file: pairs of this build and of earlier ones."""
import ctypes as C
import json
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

RUN = """
import ctypes as C, sys
sys.path[:0] = [{root!r}, {here!r}]
import workloads as W
from host_tools import load
from paper_2106_13995_gb300 import sim
out = (C.c_int * 4)()
load("program_tool").tuned(C.byref(sim.marshal(W.qft(18)).c), {dt}, out)
print(list(out))
"""


def options(tmp_path, entry, dt):
    """[fusion width, tile size, tensor cores, permutation runs] of qft(18)."""
    import workloads as W
    from host_tools import load
    load("program_tool")   # (built before the other process loads it)
    n_ops, bucket = len(W.qft(18).ops), 0
    while n_ops > 1:
        n_ops, bucket = n_ops * 8 // 9, bucket + 1
    arity = max(len(o.qubits()) for o in W.qft(18).ops)
    f = tmp_path / "tune.json"
    e = {"n": 18, "dtype": dt, "ops_bucket": bucket, "arity": arity, **entry}
    f.write_text("[\n  " + json.dumps(e) + "\n]\n")
    code = RUN.format(root=os.path.dirname(HERE), here=HERE, dt=dt)
    r = subprocess.run([sys.executable, "-c", code], env={**os.environ, "SV_TUNE_CACHE": str(f)}, check=True,
                       capture_output=True, text=True)
    return json.loads(r.stdout.splitlines()[-1])


@pytest.mark.parametrize("dt", [0, 1])
def test_pairs_of_earlier_builds_keep_the_special_paths(tmp_path, dt):
    assert options(tmp_path, {"fusion_k": 4, "tile_m": 12}, dt) == [4, 12, dt, 1]


@pytest.mark.parametrize("dt", [0, 1])
def test_pairs_that_beat_the_defaults_replace_them(tmp_path, dt):
    assert options(tmp_path, {"fusion_k": 4, "tile_m": 12, "vs_defaults": 1}, dt) == [4, 12, 0, 0]


@pytest.mark.parametrize("dt", [0, 1])
def test_defaults_that_won_stay(tmp_path, dt):
    got = options(tmp_path, {"fusion_k": 0, "tile_m": 0, "vs_defaults": 1}, dt)
    assert got[2:] == [dt, 1]
    assert got == options(tmp_path, {"fusion_k": 0, "tile_m": 0}, dt)
