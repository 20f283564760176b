"""Builds the host-side test tools that link the library's objects."""
import ctypes as C
import glob
import importlib
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def load(name):
    """tests/host/<name>.cu as a shared library next to the library's objects."""
    import paper_2106_13995_gb300 as P
    b = importlib.import_module("paper_2106_13995_gb300.buildlib")
    P.build()
    objs = sorted(glob.glob(os.path.join(b.OUT_DIR, "*.o")))
    out = os.path.join(HERE, "host", "_build")
    os.makedirs(out, exist_ok=True)
    lib, src = os.path.join(out, f"lib{name}.so"), os.path.join(HERE, "host", f"{name}.cu")
    if not os.path.exists(lib) or any(os.path.getmtime(d) > os.path.getmtime(lib) for d in [src] + objs):
        subprocess.check_call([b.nvcc(), *b.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                               "-I", os.path.join(os.path.dirname(HERE), "include"), "-o", lib, src, *objs])
    return C.CDLL(lib)
