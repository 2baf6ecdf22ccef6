"""The tile geometry of the pair and the double kernel, checked on the host:
staged cells, lines, Delta F places and face constants of every compiled tile shape
(tests/_sym_geometry.cu, built with nvcc for the host only; no GPU is used)."""
import os
import shutil
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_sym_geometry_maps():
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if nvcc is None:
        pytest.skip("nvcc not found")
    with tempfile.TemporaryDirectory() as tmp:
        exe = os.path.join(tmp, "sym_geometry")
        cmd = [nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
               "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1403_6126_gb300", "csrc"),
               os.path.join(HERE, "_sym_geometry.cu"), "-o", exe]
        b = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
        assert b.returncode == 0, b.stderr[-3000:]
        r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0 and r.stdout.strip().endswith("OK"), (r.stdout[-3000:], r.stderr[-2000:])
