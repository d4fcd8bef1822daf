"""Device headers compiled for the host with tests/device_shim.h (a C interface for ctypes)."""
import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def compile_shim(source, folder):
    """The library of tests/<source>, built in `folder` (a pathlib.Path)."""
    (folder / "cuda_runtime.h").write_text('#include "device_shim.h"\n')
    so = str(folder / "shim.so")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", str(folder), "-I", HERE,
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2110_00256_gb300", "csrc"),
                    os.path.join(HERE, source), "-o", so], check=True)
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)
