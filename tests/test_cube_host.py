"""Host-side check of the three-dimensional slab kernels' shared-memory layout
(csrc/dust_cube.cuh), compiled with nvcc as host code."""
import os
import shutil
import subprocess

import pytest

from test_host_logic import ROOT


def test_cube_shared_memory(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "cube_smem_check")
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_1908_10793_gb300", "csrc"),
                           "-gencode", "arch=compute_103a,code=sm_103a",
                           os.path.join(ROOT, "tests", "host", "cube_smem_check.cu"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
