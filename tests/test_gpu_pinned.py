"""The page-locked bytes that small reads back go through: a thread that ends
spoils no other thread's stream capture, and systems made after a device reset
do not use the bytes of the context before it.
"""
import os
import subprocess
import sys
import threading
import time

import pytest

import oracle
from paper_2408_04343_gb300 import libsnp, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_04343_gb300 import build
    build.build()
    libsnp.load()


def test_thread_that_ends_beside_another_threads_capture():
    """A thread that has waited for a result ends while this one captures a
    stream in the default (global) mode: the capture is not spoilt."""
    d = synth.random_system(900, 21, outdeg=(2, 8), rules=(2, 4), d_range=(0, 3), spikes=(0, 10))
    g = libsnp.System(d, stream=torch.cuda.Stream())
    x = torch.zeros(64, device="cuda")
    got, stepped, go = [], threading.Event(), threading.Event()

    def work():
        got.append(g.step(5))
        stepped.set()
        go.wait(30)

    t = threading.Thread(target=work)
    t.start()
    assert stepped.wait(30)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x += 1.0
        go.set()
        t.join()
        time.sleep(0.3)  # the thread's own storage goes after its Python part
        x += 1.0
    graph.replay()
    torch.cuda.synchronize()
    assert (x == 2.0).all()
    st = oracle.initial_state(d)
    assert got == [oracle.run(d, st, 5)[0]] and (g.config() == st[0]).all()
    g.close()


CHILD = """
import ctypes as ct, sys
sys.path.insert(0, sys.argv[1])
import oracle
from paper_2408_04343_gb300 import libsnp, synth
libsnp.load()
rt = ct.CDLL("libcudart.so.13")
d = synth.random_system(700, 22, outdeg=(2, 8), rules=(2, 4), d_range=(0, 3), spikes=(0, 10))
st = oracle.initial_state(d)
ex, S = oracle.run(d, st, 9)
for _ in range(3):
    g = libsnp.System(d)
    assert g.step(9) == ex
    C, D, P, k = g.get_state()
    assert k == ex and (C == st[0]).all() and (D == st[1]).all() and (P == st[2]).all()
    g.close()
    assert rt.cudaDeviceReset() == 0
print("ok")
"""


def test_systems_made_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), (r.returncode, r.stdout, r.stderr[-2000:])
