"""That the eliminated walk is what runs where its tests mean it to (by the operations
a result counts), and the two ends of its launch: up to 2,048 task results are summed
by the walk's last block, more by a reduction kernel in a replayed graph."""
import numpy as np
import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
GEN, CG = A.PERM_ENGINE_GENERIC, A.PERM_ENGINE_CODEGEN


def is_eliminated(r, a, **kw):
    return r.fp_ops_per_step < 0.6 * A.permanent(a, ordering=A.PERM_ORDER_DEGREE, **kw).fp_ops_per_step


@pytest.mark.parametrize("values", ["01", "f64"])
def test_every_call_takes_the_eliminated_walk(values):
    a = synth.single_er(24, 0.2, 41, values=values, shuffle_cols=True)
    with A.Server() as s:
        served = s.poll(s.submit(a), 60000)
    for r in (A.permanent(a), A.permanent(a, engine=GEN), A.permanent_noalloc(a), A.batch([a])[0], served):
        assert is_eliminated(r, a, engine=GEN)
    assert is_eliminated(A.permanent(a, engine=CG), a, engine=CG)


@pytest.mark.parametrize("engine,values", [(GEN, "01"), (GEN, "f64"), (CG, "01")], ids=["table_01", "table_f64", "generated_01"])
@pytest.mark.parametrize("tasks", [2047, 2048, 2049])
def test_both_sides_of_the_fused_reduction(engine, values, tasks):
    """Ranges [2^s, (tasks + 1) 2^s): the alignment lets only s columns be summed out or
    chunked, and some s gives exactly `tasks` tasks.  Three computes of one plan each."""
    n = 26
    a = synth.single_er(n, 0.3 if values == "01" else 0.4, 77, values=values)
    ao = np.ascontiguousarray(a[:, list(A.inspect(a).col_order)[:n]])
    for s in range(9, 14):
        lo, hi = 1 << s, (tasks + 1) << s
        p = A.Plan(a, engine=engine, g_lo=lo, g_hi=hi)
        r = p.compute()
        if (tasks << s) >> r.chunk_log2 == 32 * tasks:
            break
        p.close()
    else:
        raise AssertionError("no alignment gives this many tasks")
    assert is_eliminated(r, a, engine=engine, g_lo=lo, g_hi=hi)
    if values == "01":
        want = oracle.nw2_range(ao, lo, hi, threads=16)
    else:
        want, sa = oracle.nw_range(ao, lo, hi, threads=16)
    for r in (r, p.compute(), p.compute()):
        if values == "01":
            mask = (1 << (64 * min(r.exact_words, 2))) - 1
            assert r.partial_int & mask == want & mask
        else:
            assert abs((r.f64 - want.hi) + (r.f64_lo - want.lo)) <= 64 * n * U * float(sa)
            assert abs(r.abs_term_sum - float(sa)) <= 1e-4 * float(sa)
    p.close()
