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
lib.fake_fail.argtypes = [C.c_longlong, C.c_longlong]
lib.fake_solves.argtypes = [C.c_int, C.c_double]
lib.fake_live.restype = lib.fake_peak.restype = C.c_longlong
GB = 1 << 30
def counts():
    n = (C.c_int * 7)()
    lib.fake_counts(n)
    return dict(zip(("solves", "graphs", "marches", "applies", "lengths", "ng", "outside"), n))
"""


def build(folder):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")

    def sh(*cmd):
        return subprocess.run(cmd, check=True, capture_output=True, text=True, timeout=600).stdout

    api, fake, stubs = (os.path.join(folder, n) for n in ("api.o", "fake.o", "stubs.c"))
    flags = ["-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")]
    sh(nvcc, *flags, "-c", os.path.join(CSRC, "api.cu"), "-o", api)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    sh("g++", "-std=c++17", "-O1", "-w", "-fPIC", "-I", cuda, "-c",
       os.path.join(HERE, "native", "fake_device.cpp"), "-o", fake)

    def symbols(which):
        return {line.split()[-1] for o in (api, fake) for line in sh("nm", which, o).splitlines() if line.strip()}

    names = {n for n in symbols("-u") if n.startswith(("cuda", "__cuda", "_ZN4rt3d"))} | set(exported_names())
    names = sorted(names - symbols("--defined-only"))
    with open(stubs, "w") as f:
        f.writelines(f"long {n}(void) {{ return 0; }}\n" for n in names)
    lib = os.path.join(folder, "librt3d_fake.so")
    sh("gcc", "-w", "-fPIC", "-c", stubs, "-o", stubs + ".o")
    sh("g++", "-shared", "-o", lib, api, fake, stubs + ".o", "-Wl,-Bsymbolic")
    return lib


def run(lib, script, timeout=300):
    subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT, lib=lib) + script], check=True,
                   timeout=timeout)
