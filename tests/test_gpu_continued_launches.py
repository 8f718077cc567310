"""Calls of more steps than one cooperative launch takes (2^24; 7 in the
bounds-checked build, which runs here in a process of its own): the launches
that continue a call carry its start, its halt, the chosen rules and the
counters over, with every device index checked.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import numpy as np, torch
import oracle
from paper_2408_04343_gb300 import libsnp, synth
from test_zz_no_alloc import dag_system, device_tables, fresh_state

SEL = {oracle.FIRST: libsnp.SNP_SELECT_FIRST, oracle.PHILOX: libsnp.SNP_SELECT_PHILOX}
kw = dict(outdeg=(2, 9), d_range=(0, 4), spikes=(0, 10))
rand = {"records": synth.random_system(9001, 1, rules=(2, 4), **kw),
        "tests": synth.random_system(9001, 2, rules=(2, 6), k_range=(1, 40), j_range=(0, 13), **kw),
        "tables": synth.random_system(9001, 3, rules=(9, 14), k_range=(1, 12), j_range=(0, 2), **kw),
        "general": synth.random_system(9001, 4, rules=(2, 6), k_range=(1, 40), j_range=(0, 13), p_range=(1, 3000), **kw),
        "halts": dag_system(9001, 5)}

def check(what, g_step, g_state, d, mode, calls):
    st, k, S = oracle.initial_state(d), 0, np.full(d.q, -1, np.int32)
    for n in calls:
        done = g_step(k, n)
        ex, got = oracle.run(d, st, n, mode, 7, step0=k)
        assert done == ex, (what, n, done, ex)
        k, S = k + ex, got if ex else S
        C, D, P, mine = g_state()
        assert (C == st[0]).all() and (D == st[1]).all() and (P == st[2]).all() and (mine == S).all(), (what, n)

for mode in (oracle.FIRST, oracle.PHILOX):
    for name, d in rand.items():
        calls = (3, 14, 15, 40) if name == "halts" else (3, 7, 8, 22)
        for form in (libsnp.SNP_FORM_OPT, libsnp.SNP_FORM_ELL):
            if form == libsnp.SNP_FORM_ELL and name not in ("records", "halts"):
                continue
            g = libsnp.System(d, select=SEL[mode], seed=7, form=form)
            assert form == libsnp.SNP_FORM_ELL or g.info().tiled_layout == 3
            check((name, form, mode), lambda k, n: g.step(n), lambda: g.get_state()[:3] + (g.spiking(),), d, mode, calls)
            g.close()
        tabs, (C, D, P, S) = device_tables(d), fresh_state(d)
        check((name, "noalloc", mode),
              lambda k, n: libsnp.snp_step_noalloc(d.q, d.m, C=C, D=D, P=P, S=S, select=SEL[mode], seed=7, step=k, n=n, **tabs),
              lambda: tuple(x.cpu().numpy() for x in (C, D, P, S)), d, mode, calls)
print("ok")
"""


def test_calls_that_continue_in_further_launches():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_04343_gb300 import build
    build.build(check_bounds=True)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, SNP_CHECK_BOUNDS="1"))
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), (r.returncode, r.stdout, r.stderr[-3000:])
