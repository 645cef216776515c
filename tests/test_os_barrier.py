"""The barrier of the one-kernel operator-splitting solve (csrc/osbarrier.cuh),
compiled for the host and run by threads whose waits are short enough to give
up: either all of them get through the last barrier of a round or none does, so
that a solve of which one block gave up cannot report a sweep count."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_blocks_agree_whether_a_wait_gave_up(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "os_barrier")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-pthread", "-o", exe,
                    os.path.join(HERE, "native", "os_barrier.cu")],
                   check=True, capture_output=True, timeout=300)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=240).stdout
    passed, gone, disagreed, wrong = map(int, out.split())
    assert passed > 1000 and gone > 100
    assert disagreed == 0 and wrong == 0
