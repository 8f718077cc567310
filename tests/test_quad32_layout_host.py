"""The grid-resident engine's in-lists, decoded on the CPU (no GPU): every neuron's
list holds exactly its in-neighbours, by word and bit in the packed emissions, at
every width; pads and slack name the place past the last group.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2408_04343_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("quads32") / "quad32_layout_check")
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                        os.path.join(ROOT, "tests", "quad32_layout_check.cpp"), os.path.join(CSRC, "pack.cpp"),
                        "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


@pytest.mark.parametrize("q,deg", [(1, 0), (5, 4), (127, 9), (128, 9), (130, 9), (1000, 30), (8195, 5), (70001, 6)])
@pytest.mark.parametrize("bits", [2, 4, 8, 16])
def test_lists_decode_to_the_in_lists(checker, q, deg, bits):
    r = subprocess.run([checker, str(q), str(deg), str(q + deg), str(bits)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr[-2000:])
