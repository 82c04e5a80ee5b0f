"""The slot lists of the trajectory recursion, run on the host (no GPU) against
dense products (tests/host/ric_schedule.cu)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_recursion_schedules_match_dense_products_on_host(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "ric_schedule")
    cmd = [nvcc, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"),
           "-I", os.path.join(ROOT, "paper_2406_07048_gb300", "csrc"), "-o", exe,
           os.path.join(ROOT, "tests", "host", "ric_schedule.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    print(out.stdout)
    assert out.returncode == 0, out.stdout
    seen = {tuple(int(v) for v in line.split()[:2]) for line in out.stdout.split("\n") if line.strip()}
    assert seen == {(0, 16), (0, 32), (1, 16), (1, 32), (2, 128)}
