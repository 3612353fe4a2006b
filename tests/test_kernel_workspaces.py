"""Launch shapes and shared-memory workspaces of the polish over active neurons
and of the sparse re-decision (host arithmetic only, no GPU): for every layer
width, input dimension, sign-word count and number of parameters, in both builds
(`tests/c/kernel_workspaces.cu` includes the kernel sources as they are)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("max_d", [8, 10])
def test_kernel_workspaces(tmp_path, max_d):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / f"kernel_workspaces_{max_d}")
    cmd = [nvcc, "-std=c++17", f"-DPC_MAX_D={max_d}", "-gencode", "arch=compute_103a,code=compute_103a", "-Xcicc", "-O0",
           "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_2306_07212_gb300", "csrc"),
           os.path.join(ROOT, "tests", "c", "kernel_workspaces.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("0 failures"), r.stdout[-2000:]
