"""The double kernel's reciprocal and quotient against CUDA's division
(tests/_rcp_double.cu, built with nvcc and run on the GPU)."""
import os
import subprocess

import pytest

from paper_1403_6126_gb300 import build as rtbuild

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_reciprocal_matches_division(tmp_path):
    exe = str(tmp_path / "rcp_double")
    subprocess.check_call([rtbuild.NVCC] + rtbuild.ARCH + ["-O3", "-std=c++17", "-I", rtbuild.INCLUDE, "-I", rtbuild.CSRC,
                                                           os.path.join(HERE, "_rcp_double.cu"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("OK"), (r.stdout, r.stderr)
