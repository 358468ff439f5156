"""The cluster factor's launch on every device of a process (csrc/
chol_cluster.cu): a kernel's permission for clusters of more than 8 CTAs, and
whether one can be placed, belong to a device.  The library's object is run
against a stand-in for the CUDA runtime (tests/emu/chol_host.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_each_device_gets_a_cluster_that_it_takes(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    from paper_2609_00049_gb300 import build as b
    b.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(b.nvcc())))
    exe = str(tmp_path / "chol_host")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", b.CSRC, "-I", b.INCLUDE, "-I", os.path.join(cuda, "include"),
                    os.path.join(ROOT, "tests", "emu", "chol_host.cpp"), os.path.join(b.BUILD, "chol_cluster.o"),
                    "-o", exe, "-lpthread"], check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout
    got = [tuple(map(int, line.split())) for line in out.splitlines()]
    want = [(dev, vec, 0, 8 if dev == 2 else 16) for _ in range(2) for dev in range(3) for vec in range(2)]
    assert got == want
