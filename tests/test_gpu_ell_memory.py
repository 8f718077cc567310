"""The ELL form's device memory: systems stepped on one-word pairs hold no vectors
of emitting rules beside the bits.
"""
import dataclasses

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


def with_forgetting_rules(d, extra):
    """`extra` more forgetting rules at the end of every neuron."""
    R = np.diff(d.rule_offsets)
    at = np.repeat(d.rule_offsets[1:], extra)
    ins = lambda a, v: np.insert(a, at, np.int32(v))
    return dataclasses.replace(d, rule_offsets=np.concatenate([[0], np.cumsum(R + extra)]), rule_k=ins(d.rule_k, 3),
                               rule_j=ins(d.rule_j, 0), rule_c=ins(d.rule_c, 3), rule_p=ins(d.rule_p, 0),
                               rule_d=ins(d.rule_d, 0))


def test_a_rule_costs_its_word_only():
    d = synth.random_system(20_000, 3, outdeg=(2, 8), rules=(2, 2), d_range=(0, 3), spikes=(0, 10))
    held = []
    for extra in (0, 2):
        g = libsnp.System(with_forgetting_rules(d, extra), form=libsnp.SNP_FORM_ELL)
        g.step(3)
        held.append(g.info().device_bytes)
        g.close()
    per_rule = (held[1] - held[0]) / (2 * d.q)
    assert per_rule < 4.1, per_rule
