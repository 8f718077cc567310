"""Paths that only extreme or simultaneous systems take: a push whose in-flow could
leave 32 bits (added to the counts directly), the ELL pull of more neurons than
the bit vector holds, two grid-resident systems stepped from two threads.
"""
import threading

import numpy as np
import pytest

import oracle
from paper_2408_04343_gb300 import libsnp, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SEL = {oracle.FIRST: libsnp.SNP_SELECT_FIRST, oracle.PHILOX: libsnp.SNP_SELECT_PHILOX}


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_04343_gb300 import build
    build.build()
    libsnp.load()


def same(g, d, st, S):
    C, D, P, _ = g.get_state()
    assert (C == st[0]).all() and (D == st[1]).all() and (P == st[2]).all()
    assert (g.spiking() == S).all()


@pytest.mark.parametrize("form", [libsnp.SNP_FORM_OPT, libsnp.SNP_FORM_ELL])
@pytest.mark.parametrize("mode", [oracle.FIRST, oracle.PHILOX])
def test_push_whose_in_flow_could_leave_32_bits(form, mode):
    q = 45_000
    d = synth.random_system(q, 11, outdeg=(2, 6), rules=(2, 4), d_range=(0, 3), spikes=(0, 10))
    hub = 17  # every neuron sends to it; one rule that seldom applies sends 65,535
    rows = [d.syn_targets[d.syn_offsets[i]:d.syn_offsets[i + 1]] for i in range(q)]
    rows = [t if i == hub or hub in t else np.append(t, np.int32(hub)) for i, t in enumerate(rows)]
    d.syn_targets = np.concatenate(rows).astype(np.int32)
    d.syn_offsets = np.concatenate([[0], np.cumsum([len(t) for t in rows])]).astype(np.int64)
    d.rule_p[int(d.rule_offsets[100])] = 65_535
    g = libsnp.System(d, select=SEL[mode], seed=4, form=form, prop=libsnp.SNP_PROP_PUSH)
    st, k = oracle.initial_state(d), 0
    for n in (1, 8):
        assert g.step(n) == n
        ex, S = oracle.run(d, st, n, mode, 4, step0=k)
        k += ex
        assert ex == n
        same(g, d, st, S)
    g.close()


def test_ell_pull_of_more_neurons_than_the_bits_hold():
    d = synth.random_system(409_601, 12, outdeg=(1, 4), rules=(2, 3), d_range=(0, 3), spikes=(0, 10))
    g = libsnp.System(d, select=libsnp.SNP_SELECT_PHILOX, seed=4, form=libsnp.SNP_FORM_ELL)
    st = oracle.initial_state(d)
    ex, S = oracle.run(d, st, 5, oracle.PHILOX, 4)
    assert g.step(5) == ex
    same(g, d, st, S)
    g.close()


def test_two_grid_resident_systems_from_two_threads():
    descs = [synth.random_system(q, q, outdeg=(2, 8), rules=(2, 4), d_range=(0, 3), spikes=(0, 10)) for q in (30_011, 90_001)]
    systems = [libsnp.System(d, select=libsnp.SNP_SELECT_PHILOX, seed=6, stream=torch.cuda.Stream()) for d in descs]
    assert all(g.info().tiled_layout == 3 for g in systems)
    done, failed = [0, 0], []

    def work(i):
        try:
            for _ in range(20):
                done[i] += systems[i].step(6)
        except Exception as e:  # noqa: BLE001 -- reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for g, d, n in zip(systems, descs, done):
        st = oracle.initial_state(d)
        ex, S = oracle.run(d, st, 120, oracle.PHILOX, 6)
        assert n == ex == 120
        C, D, P, k = g.get_state()
        assert k == 120
        assert (C == st[0]).all() and (D == st[1]).all() and (P == st[2]).all()
        g.close()
