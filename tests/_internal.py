"""Builds internal_entry.cpp against the library and loads it."""
import ctypes
import os
import subprocess

from _gpu_common import built_package

HERE = os.path.dirname(os.path.abspath(__file__))


def internal():
    P = built_package()
    src, out = os.path.join(HERE, "internal_entry.cpp"), os.path.join(HERE, "_build", "internal_entry.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    csrc, lib = os.path.join(os.path.dirname(HERE), "paper_1808_07217_gb300", "csrc"), P.LIB_PATH
    if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(p) for p in (src, lib)):
        tmp = f"{out}.{os.getpid()}"
        subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", "/usr/local/cuda/include", "-I", csrc, src,
                        "-o", tmp, "-L", os.path.dirname(lib), "-l:" + os.path.basename(lib),
                        "-Wl,-rpath," + os.path.dirname(lib)], check=True)
        os.replace(tmp, out)
    return ctypes.CDLL(out)


def ptr(t):
    return ctypes.c_void_p(0 if t is None else t.data_ptr())
