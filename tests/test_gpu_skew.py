"""AUTO's middle sizes with long in-lists: a system whose longest lists would keep
one warp of the grid-resident engine busy takes the tiled engine's launch per
step, and results on either side of that line equal the oracle's -- alone and
in a batch, which keeps its own lists of such systems.
"""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2408_04343_gb300 import libsnp, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SEL = {oracle.FIRST: libsnp.SNP_SELECT_FIRST, oracle.PHILOX: libsnp.SNP_SELECT_PHILOX}
GRID_LAYOUT = 3  # snp_info.tiled_layout


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_04343_gb300 import build
    build.build()
    libsnp.load()


def with_in_degrees(q, seed, deg, **kw):
    """A random system in which neuron t has about deg[t] in-edges."""
    rng = np.random.default_rng(seed)
    d = synth.random_system(q, seed, outdeg=(0, 0), **kw)
    t = np.repeat(np.arange(q, dtype=np.int64), np.minimum(deg, q - 1))
    s = rng.integers(0, q - 1, size=t.size)
    s += s >= t
    key = np.unique(s * q + t)
    off = np.zeros(q + 1, np.int64)
    np.cumsum(np.bincount(key // q, minlength=q), out=off[1:])
    return dataclasses.replace(d, syn_offsets=off, syn_targets=(key % q).astype(np.int32))


RULES = {"records": dict(rules=(2, 4)), "tests": dict(rules=(2, 6), k_range=(1, 40), j_range=(0, 13)),
         "tables": dict(rules=(9, 14), k_range=(1, 12), j_range=(0, 2))}


# a hub's list, and whether one launch still runs all steps: short enough for
# shared memory, walked by several warps, too long; with and without quads
# kept for batches (65,536 neurons)
@pytest.mark.parametrize("q,hub,rules,grid", [(9001, 200, "records", True), (9001, 3000, "records", False),
                                              (40_003, 200, "records", True), (40_003, 30_000, "records", False),
                                              (40_003, 1200, "tests", True), (40_003, 12_000, "tests", False),
                                              (40_003, 12_000, "tables", False), (90_001, 12_000, "records", False)])
def test_one_hub(q, hub, rules, grid):
    deg = np.random.default_rng(q).integers(4, 12, size=q)
    deg[q // 3] = hub
    d = with_in_degrees(q, 90 + q, deg, d_range=(0, 4), spikes=(0, 10), **RULES[rules])
    for mode in (oracle.FIRST, oracle.PHILOX):
        g = libsnp.System(d, select=SEL[mode], seed=5)
        assert (g.info().tiled_layout == GRID_LAYOUT) == grid
        assert g.info().engine == libsnp.SNP_ENGINE_TILED
        st, k = oracle.initial_state(d), 0
        for n in (1, 11):
            assert g.step(n) == n
            ex, S = oracle.run(d, st, n, mode, 5, step0=k)
            k += n
            C, D, P, _ = g.get_state()
            assert ex == n and (C == st[0]).all() and (D == st[1]).all() and (P == st[2]).all()
            assert (g.spiking() == S).all()
        g.close()


def test_power_law_in_degrees_alone_and_in_a_batch():
    q = 20_000
    w = np.arange(1, q + 1) ** -0.8
    deg = np.random.default_rng(1).permutation(np.maximum(1, w / w.sum() * 8 * q).astype(np.int64))
    d = with_in_degrees(q, 17, deg, rules=(2, 4), d_range=(0, 4), spikes=(0, 10))
    alone = libsnp.System(d, select=libsnp.SNP_SELECT_PHILOX, seed=8)
    assert alone.info().tiled_layout != GRID_LAYOUT
    member = libsnp.System(d, select=libsnp.SNP_SELECT_PHILOX, seed=8, deferred=True)
    b = libsnp.Batch()
    st = oracle.initial_state(d)
    ex, S = oracle.run(d, st, 70, oracle.PHILOX, 8)
    assert alone.step(70) == ex and b.wait(b.submit([member], 70)) == [ex]
    for g in (alone, member):
        C, D, P, k = g.get_state()
        assert k == ex and (C == st[0]).all() and (D == st[1]).all() and (P == st[2]).all()
        assert (g.spiking() == S).all()
        g.close()
    b.close()
