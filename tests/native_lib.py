"""Builds a source of tests/native against the library and loads it."""
import ctypes
import os
import subprocess

from paper_2210_03699_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def load(name):
    lib = build.build()
    src = os.path.join(HERE, "native", name)
    out = os.path.join(build.OUT_DIR, f"libtest_{name.split('.')[0]}.so")
    if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(src), os.path.getmtime(lib)):
        tmp = out + f".tmp{os.getpid()}"
        subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC",
                        "-I", build.INCLUDE, "-I", build.SRC_DIR, src, lib, "-o", tmp], check=True)
        os.replace(tmp, out)
    return ctypes.CDLL(out)
