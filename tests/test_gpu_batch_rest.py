"""Systems of a batch that no cluster holds -- wide emissions, or more than 65,408
neurons -- made under AUTO: they run beside the others, a CTA each with packed
emissions, and equal the oracle.
"""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("mode", [oracle.FIRST, oracle.PHILOX])
def test_systems_that_fit_no_cluster(mode):
    kw = dict(outdeg=(2, 9), d_range=(0, 4), spikes=(0, 10))
    wide = dict(p_range=(1, 900), rules=(2, 4))
    descs = [synth.random_system(50_001, 1, **kw, **wide), synth.random_system(65_409, 2, rules=(2, 4), **kw),
             synth.random_system(65_536, 3, rules=(3, 3), p_range=(1, 40), **kw),
             synth.random_system(56_000, 4, **kw, **wide)]
    small = [synth.random_system(700, 5, rules=(2, 4), **kw), synth.random_system(30_000, 6, **kw, **wide)]
    select = libsnp.SNP_SELECT_FIRST if mode == oracle.FIRST else libsnp.SNP_SELECT_PHILOX
    make = lambda ds: [libsnp.System(d, select=select, seed=3, deferred=True) for d in ds]
    # alone in a batch: nothing is stepped grid-wide
    b = libsnp.Batch()
    first = make(descs)
    done = [b.wait(b.submit(first, 70))]
    assert b.info().resident_device_seconds > 0
    mixed = make(descs + small)
    done.append(b.wait(b.submit(mixed, 70)))
    for systems, ds, ex in ((first, descs, done[0]), (mixed, descs + small, done[1])):
        for g, d, n in zip(systems, ds, ex):
            st = oracle.initial_state(d)
            m, S = oracle.run(d, st, 70, mode, 3)
            C, D, P, k = g.get_state()
            assert n == m == k
            assert (C == st[0]).all() and (D == st[1]).all() and (P == st[2]).all()
            assert (g.spiking() == S).all()
            # and alone afterwards, on the engine of its own
            assert g.step(5) == oracle.run(d, st, 5, mode, 3, step0=k)[0]
            assert (g.config() == st[0]).all()
            g.close()
    b.close()
