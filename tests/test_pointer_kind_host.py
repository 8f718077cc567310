"""The decision that lets snp_set_state read the caller's arrays in place, on
made-up pointer attributes (no GPU): only memory of the system's own device;
another GPU's, page-locked and plain host memory are copied.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2408_04343_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


def test_only_the_systems_own_device_is_read_in_place(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    exe = str(tmp_path / "pointer_kind_check")
    r = subprocess.run([cxx, "-O1", "-std=c++17", "-I", CUDA, "-I", CSRC,
                        os.path.join(ROOT, "tests", "pointer_kind_check.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
