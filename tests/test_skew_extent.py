"""Extents near 2^31 rows: which of them the skewed tiles take, and that their
32-bit row arithmetic holds for those (tests/skew_extent.cu, on the CPU)."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_extents_on_host(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc"
                                    if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "skew_extent")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "-I",
           os.path.join(ROOT, "paper_2604_22242_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
           os.path.join(HERE, "skew_extent.cu"), "-o", exe]
    p = subprocess.run(cmd, capture_output=True, text=True)
    assert p.returncode == 0, p.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    m = re.match(r"checked (\d+) bad 0$", r.stdout.strip())
    assert m and int(m[1]) > 10000, r.stdout
