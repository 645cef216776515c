"""The library's host code (csrc/api.cu) on a device in host memory
(native/fake_device.cpp), for tests of budgets, failed allocations and waits that gave
up.  build() makes the shared library, run() executes a script on it in a
process of its own."""

import os
import shutil
import subprocess
import sys

import pytest

from paper_1107_5719_gb300.rt3d import exported_names

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1107_5719_gb300", "csrc")

PRELUDE = """
import ctypes as C, sys
import numpy as np
sys.path.insert(0, {root!r})
from paper_1107_5719_gb300 import rt3d as R, workloads as W
lib = R.load({lib!r})
lib.fake_memory.argtypes = [C.c_longlong]
lib.fake_operator.argtypes = [C.c_int, C.c_int, C.c_ulonglong]
lib.fake_solves.argtypes = [C.c_int, C.c_double]
lib.fake_large.argtypes = [C.c_longlong]
lib.fake_live.restype = lib.fake_peak.restype = lib.fake_large.restype = C.c_longlong
GB = 1 << 30
up = lambda b: (b + 255) // 256 * 256

def rays(p):
    # bytes of a ray-by-ray recording of p in FP64 or double-float
    N, D, nxy = p.nvox, p.ndir, p.nx * p.ny
    return up(4 * D * nxy * p.nz * (p.nz - 1)) + up(4 * D * p.nz * ((nxy + 31) // 32)) + 2 * up(64 * N)

def counts():
    n = (C.c_int * 10)()
    lib.fake_counts(n)
    return dict(zip(("solves", "graphs", "marches", "applies", "lengths", "ng", "outside", "replays", "chunks", "mallocs"), n))
"""


def sh(*cmd):
    return subprocess.run(cmd, check=True, capture_output=True, text=True, timeout=600).stdout


def nvcc():
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        pytest.skip("nvcc not available")
    return path


def compile_cpp(name, obj):
    """native/<name> against the CUDA headers alone."""
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    sh("g++", "-std=c++17", "-O1", "-w", "-fPIC", "-I", cuda, "-c", os.path.join(HERE, "native", name), "-o", obj)
    return obj


def stubs(objs, folder, also=()):
    """Functions that return 0 for the CUDA calls and launches (and `also`) that
    the objects call and none of them defines."""
    def symbols(which):
        return {line.split()[-1] for o in objs for line in sh("nm", which, o).splitlines() if line.strip()}

    names = {n for n in symbols("-u") if n.startswith(("cuda", "__cuda", "_ZN4rt3d"))} | set(also)
    src = os.path.join(folder, "stubs.c")
    with open(src, "w") as f:
        f.writelines(f"long {n}(void) {{ return 0; }}\n" for n in sorted(names - symbols("--defined-only")))
    sh("gcc", "-w", "-fPIC", "-c", src, "-o", src + ".o")
    return src + ".o"


def build(folder):
    api = os.path.join(folder, "api.o")
    sh(nvcc(), "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-c",
       os.path.join(CSRC, "api.cu"), "-o", api)
    objs = [api, compile_cpp("fake_device.cpp", os.path.join(folder, "fake.o"))]
    lib = os.path.join(folder, "librt3d_fake.so")
    sh("g++", "-shared", "-o", lib, *objs, stubs(objs, folder, exported_names()), "-Wl,-Bsymbolic")
    return lib


def run(lib, script, timeout=300):
    subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT, lib=lib) + script], check=True,
                   timeout=timeout)
