"""snp_set_state from device arrays that another stream still writes: whatever it
takes in has been checked.
"""
import numpy as np
import pytest

from paper_2408_04343_gb300 import libsnp, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_04343_gb300 import build
    build.build()
    libsnp.load()


@pytest.mark.parametrize("q", [257, 60_000])
def test_every_state_taken_in_was_checked(q):
    """P alternates between -1 and a rule that does not exist while the calls
    run: a call may refuse, but a state it accepts holds no such rule."""
    d = synth.random_system(q, 5 + q, outdeg=(1, 4), rules=(3, 3), d_range=(0, 3), spikes=(0, 9))
    g = libsnp.System(d, engine=libsnp.SNP_ENGINE_LAUNCH)
    C = torch.from_numpy(d.init_spikes).cuda()
    D, P = torch.zeros_like(C), torch.full_like(C, -1)
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        for _ in range(1000):
            P.fill_(d.m + 5)
            P.fill_(-1)
    taken = refused = 0
    for _ in range(6):
        with torch.cuda.stream(side):
            for _ in range(3):
                graph.replay()
            done = torch.cuda.Event()
            done.record()
        while not done.query():
            try:
                g.set_state(C, D, P, 3)
            except libsnp.SnpError as e:
                assert e.status == libsnp.SNP_ERR_INVALID
                refused += 1
                continue
            taken += 1
            assert (g.pending() == -1).all(), (taken, refused)
    side.synchronize()
    g.set_state(C, D, P, 3)
    assert (g.config() == d.init_spikes).all() and (g.pending() == -1).all() and (g.spiking() == -1).all()
    print("taken", taken, "refused", refused)
    g.close()
