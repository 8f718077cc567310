"""snp_step_noalloc at the ends of what it accepts: in-neighbour lists that end
at entry INT32_MAX and rules at the last id, where an index plus a stride no
longer fits 32 bits.  State and executed steps equal the oracle's.
"""
import ctypes as ct

import numpy as np
import pytest

import oracle
from paper_2408_04343_gb300 import libsnp, synth
from test_zz_no_alloc import device_tables, fresh_state

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


def call_on(sms, cap, d, tabs, C, D, P, S, select, seed, step, n):
    """snp_step_noalloc as on a device of sms SMs with cap bytes of shared memory."""
    fn = libsnp.load().snp_noalloc_on
    p = lambda t: t.data_ptr()
    s = libsnp.snp_device_system(d.q, d.m, tabs["in_sources"].numel(), *(p(tabs[k]) for k in (
        "rule_offsets", "rule_k", "rule_j", "rule_c", "rule_p", "rule_d", "in_offsets", "in_sources")),
        p(C), p(D), p(P), p(S))
    done = ct.c_int64(0)
    rc = fn(ct.byref(s), ct.c_int32(select), ct.c_uint64(seed), ct.c_uint64(step), ct.c_int64(n), None,
            ct.byref(done), ct.c_int32(sms), ct.c_int32(cap))
    return rc, int(done.value)


# (SMs, shared memory): no cooperative launches; 18 SMs cannot hold 200,000
# neurons' state; 100 KB hold 4 SMs' share of 9,000; few rules and lists staged
@pytest.mark.parametrize("q,sms,cap", [(9000, 0, 0), (200_000, 18, 232448), (9000, 4, 102400), (9000, 3, 102400),
                                       (3000, 9, 14_000), (1, 1, 232448)])
@pytest.mark.parametrize("mode", [oracle.FIRST, oracle.PHILOX])
def test_devices_that_hold_less(q, sms, cap, mode):
    d = synth.random_system(q, 70 + q, outdeg=(min(2, q - 1), min(9, q - 1)), rules=(2, 6), d_range=(0, 3),
                            spikes=(0, 10))
    tabs = device_tables(d)
    C, D, P, S = fresh_state(d)
    st, k = oracle.initial_state(d), 0
    select = libsnp.SNP_SELECT_FIRST if mode == oracle.FIRST else libsnp.SNP_SELECT_PHILOX
    for n in (1, 7, 40):
        rc, done = call_on(sms, cap, d, tabs, C, D, P, S, select, 11, k, n)
        ex, S_ref = oracle.run(d, st, n, mode, 11, step0=k)
        assert rc == 0 and done == ex
        k += ex
        assert (C.cpu().numpy() == st[0]).all() and (D.cpu().numpy() == st[1]).all()
        assert (P.cpu().numpy() == st[2]).all()
        assert not ex or (S.cpu().numpy() == S_ref).all()
    C[q // 2] = -1  # checked on every form
    assert call_on(sms, cap, d, tabs, C, D, P, S, select, 11, k, 2)[0] == libsnp.SNP_ERR_INVALID
