"""GPU parity of the eliminated walk against the oracle: the generated kernel
and the precompiled one, as plans, in batches, served and without allocation,
at the edges of their ranges (the smallest n, both sides of the sizes where a
rule changes, programs of one and of several tables, rings of 2 to 6 limbs,
sub-ranges).  Exact results bit for bit; FP64 within 1e-9 of the permanent or
64 n 2^-53 of a range's sum of |terms|; double-double within its own bound."""
import numpy as np
import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
MASK128 = (1 << 128) - 1


def check(a, r):
    n = a.shape[0]
    if a.dtype == np.int64:
        assert r.value == (oracle.ryser_gray(a) if n <= 20 else oracle.rowdp_int(a))
    else:
        want = float(oracle.nw_perm(a, threads=16)[0]) if n <= 20 else float(oracle.rowdp(a))
        assert abs(r.value - want) <= 1e-9 * abs(want), (n, r.value, want)


@pytest.mark.parametrize("values", ["01", "f64"])
@pytest.mark.parametrize("n,p", [(9, 0.5), (10, 0.2), (13, 0.4), (18, 0.3), (19, 0.3), (20, 0.15), (22, 0.2), (25, 0.15),
                                 (29, 0.12), (31, 0.1), (33, 0.08)])
def test_whole_walks_on_every_path(n, p, values):
    a = synth.single_er(n, p, 40 + n, values=values, shuffle_cols=True)
    check(a, A.permanent(a))
    check(a, A.permanent(a, engine=A.PERM_ENGINE_GENERIC))
    check(a, A.permanent(a, engine=A.PERM_ENGINE_CODEGEN))
    check(a, A.permanent_noalloc(a))
    b = synth.single_er(n + 1, p, 90 + n, values=values)
    for m, r in zip([a, b, a], A.batch([a, b, a])):
        check(m, r)
    with A.Server() as s:
        for m, t in [(m, s.submit(m)) for m in (a, b)]:
            check(m, s.poll(t, 60000))


@pytest.mark.parametrize("words", [0, 1, 2, 3])
@pytest.mark.parametrize("top", [1, 3])
def test_rings_of_every_width(words, top):
    g = np.random.default_rng(7 + top)
    a = synth.single_er(21, 0.18, 5, values="01") * (g.integers(1, top + 1, (21, 21)) * g.choice([-1, 1], (21, 21)))
    want = oracle.rowdp_int(a)
    for engine in (A.PERM_ENGINE_GENERIC, A.PERM_ENGINE_CODEGEN):
        if words == 1 and A.inspect(a).exact_words > 1:
            continue
        assert A.permanent(a, engine=engine, exact_words=words).value == want


@pytest.mark.parametrize("n", [9, 16, 21])
def test_double_double(n):
    g = np.random.default_rng(n)
    a = synth.single_er(n, 0.25, n, values="f64") * g.choice([-1.0, 1.0], (n, n))
    want, sa = oracle.nw_perm(a, threads=8)
    r = A.permanent(a, precision=A.PERM_PREC_DD)
    tol = 64 * n * (2.0 ** -104 + 2.0 ** -oracle.long_double_bits()) * float(sa)
    assert abs((r.f64 - want.hi) + (r.f64_lo - want.lo)) <= tol
    assert abs(r.abs_term_sum - float(sa)) <= 1e-5 * float(sa)


@pytest.mark.parametrize("engine", [A.PERM_ENGINE_GENERIC, A.PERM_ENGINE_CODEGEN])
@pytest.mark.parametrize("values", ["01", "f64"])
def test_sub_ranges_keep_the_plans_partial_sums(engine, values):
    """Ranges of 2^17, 2^20 + 2^17 and 2^22 steps at several offsets: every
    position below the range's alignment may be summed out, none above it."""
    a = synth.band_plus(40, 2, 1, seed=4, values=values)
    plan = np.ascontiguousarray(a[:, list(A.inspect(a).col_order)[:40]])
    for lo, hi in ((0, 1 << 17), (1 << 33, (1 << 33) + (9 << 17)), (5 << 22, 6 << 22), ((1 << 39) - (1 << 22), 1 << 39)):
        r = A.permanent(a, g_lo=lo, g_hi=hi, engine=engine, flags=A.PERM_FLAG_ABS_SUM)
        if values == "01":
            assert r.partial_int & MASK128 == oracle.nw2_range(plan, lo, hi, threads=16)
        else:
            s, sa = oracle.nw_range(plan, lo, hi, threads=16)
            assert abs(r.value - float(s)) <= 64 * 40 * U * float(sa)
            assert abs(r.abs_term_sum - float(sa)) <= 1e-5 * float(sa)
