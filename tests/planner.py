"""Builds tests/native/planner.cpp against the library and loads it."""
import ctypes
import os
import subprocess

from paper_2210_03699_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def load():
    lib = build.build()
    src = os.path.join(HERE, "native", "planner.cpp")
    out = os.path.join(build.OUT_DIR, "libtest_planner.so")
    if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(src), os.path.getmtime(lib)):
        tmp = out + f".tmp{os.getpid()}"
        subprocess.run([build._nvcc(), "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC", "-I", build.INCLUDE,
                        "-I", build.SRC_DIR, src, lib, "-o", tmp], check=True)
        os.replace(tmp, out)
    P = ctypes.CDLL(out)
    for f in ("plan_direct", "plan_tree"):
        getattr(P, f).restype = ctypes.c_int64
    return P
