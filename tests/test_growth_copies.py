"""The copies of growing buffers and of results: none asks cudaMemcpy2DAsync for
a pitch above its limit of 2^31 - 1 bytes (values lie vertex by vertex, so their
one row is the whole buffer), every range lies in its buffer and none is left
out (`tests/c/growth_copies.cu` includes the host code and records the copies)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_growth_copies(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    from paper_2306_07212_gb300 import buildlib
    buildlib.build()  # the other sources' entry points
    exe = str(tmp_path / "growth_copies")
    cmd = [nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=compute_103a", "-Xcicc", "-O0",
           "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_2306_07212_gb300", "csrc"),
           os.path.join(ROOT, "tests", "c", "growth_copies.cu"), buildlib.LIB,
           "-Xlinker", "-rpath," + os.path.dirname(buildlib.LIB), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("0 failures"), r.stdout[-2000:]
