"""snp_step_noalloc at the ends of what it accepts: in-neighbour lists that end
at entry INT32_MAX and rules at the last id, where an index plus a stride no
longer fits 32 bits.  State and executed steps equal the oracle's.
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


def unit_rules(d):
    """The system with one rule a -> a;0 in every neuron."""
    one, zero = np.ones(d.q, np.int32), np.zeros(d.q, np.int32)
    return synth.SystemDesc(q=d.q, init_spikes=d.init_spikes, rule_offsets=np.arange(d.q + 1, dtype=np.int64),
                            rule_k=one, rule_j=zero, rule_c=one, rule_p=one, rule_d=zero,
                            syn_offsets=d.syn_offsets, syn_targets=d.syn_targets)


@pytest.mark.parametrize("q", [1, 5, 700])
def test_lists_and_rules_at_the_ends_of_the_largest_arrays(q):
    last = 2**31 - 1
    if torch.cuda.mem_get_info()[0] < 30 * 2**30:
        pytest.skip("needs 26 GB of device memory")
    d = unit_rules(synth.random_system(q, 60 + q, outdeg=(min(1, q - 1), min(9, q - 1)), spikes=(0, 2)))
    src = np.repeat(np.arange(q, dtype=np.int64), np.diff(d.syn_offsets))
    order = np.argsort(d.syn_targets, kind="stable")
    off = np.zeros(q + 1, np.int64)
    np.cumsum(np.bincount(d.syn_targets, minlength=q), out=off[1:])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()
    m = last - 1
    ones = torch.ones(m, dtype=torch.int32, device="cuda")
    zeros = torch.zeros(m, dtype=torch.int32, device="cuda")
    lists = torch.zeros(last, dtype=torch.int32, device="cuda")
    if src.size:
        lists[-src.size:] = dev(src[order])
    C, D = dev(d.init_spikes), torch.zeros(q, dtype=torch.int32, device="cuda")
    P, S = (torch.full((q,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    done = libsnp.snp_step_noalloc(q, m, dev(m - q + np.arange(q + 1)), ones, zeros, ones, ones, zeros,
                                   dev(last - src.size + off), lists, C, D, P, S, n=12)
    st = oracle.initial_state(d)
    ex, S_ref = oracle.run(d, st, 12, oracle.FIRST, 0)
    assert done == ex
    assert (C.cpu().numpy() == st[0]).all() and (D.cpu().numpy() == 0).all() and (P.cpu().numpy() == -1).all()
    if ex:
        assert (S.cpu().numpy() == np.where(S_ref >= 0, S_ref + (m - q), -1)).all()
