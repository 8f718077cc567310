"""Packing the quad lists takes time in proportion to their entries, also where a
list's sources share a bank (a search of the list per entry took 100 times as
long there).
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2408_04343_gb300", "csrc")


def test_sources_of_one_bank_pack_as_fast_as_mixed_ones(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "pack_time_check")
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                        os.path.join(ROOT, "tests", "pack_time_check.cpp"), os.path.join(CSRC, "pack.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
    mixed, shared = map(float, r.stdout.split())
    assert shared < 12 * mixed, (mixed, shared)
