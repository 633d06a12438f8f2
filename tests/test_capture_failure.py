"""Host state after a kernel launch that returns an error, in a step and while
a batch's steps are being captured: the library's objects linked with a CUDA
runtime of host functions (no GPU; see tests/host/capture_failure_check.cpp)."""
import os
import shutil
import subprocess

import pytest

from paper_1908_10793_gb300 import build
from test_host_logic import ROOT, _cuda_include


def test_failed_launches_leave_no_stale_clears(tmp_path):
    cxx, inc = shutil.which("g++"), _cuda_include()
    if cxx is None or inc is None or not os.path.exists(build._nvcc()):
        pytest.skip("g++ or CUDA not available")
    build.build_library()
    objects = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    if not all(os.path.exists(o) for o in objects):
        build.build_library(force=True)
    exe = str(tmp_path / "capture_failure_check")
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", inc,
                           os.path.join(ROOT, "tests", "host", "capture_failure_check.cpp")] + objects + ["-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
