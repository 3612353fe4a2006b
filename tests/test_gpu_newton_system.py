"""The Newton solve of the FP64 sign re-decision on ill-conditioned systems
(nearly parallel zero sets): as accurate as an elimination in float64, or done
by one (`tests/c/newton_system.cu` launches newton_warp itself)."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("max_d", [8, 10])
def test_step_is_float64_accurate(tmp_path, max_d):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / f"newton_system_{max_d}")
    cmd = [nvcc, "-O3", "-std=c++17", f"-DPC_MAX_D={max_d}", "-gencode", "arch=compute_103a,code=sm_103a",
           "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_2306_07212_gb300", "csrc"),
           os.path.join(ROOT, "tests", "c", "newton_system.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0 and r.stdout.strip().endswith("0 failures"), r.stdout[-2000:]
