"""No C++ exception leaves the calls that need no host memory when there is none
(tests/_no_throw.cpp, linked with the library and run on the GPU)."""
import os
import subprocess

import pytest

from paper_1403_6126_gb300 import build as rtbuild

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_calls_without_host_memory(tmp_path):
    lib = rtbuild.build()
    exe = str(tmp_path / "no_throw")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", rtbuild.INCLUDE, os.path.join(HERE, "_no_throw.cpp"), lib,
                           "-Wl,-rpath," + os.path.dirname(lib), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("OK"), (r.stdout, r.stderr)
