"""Precision AUTO: the double-double rerun of a plan is planned like a double-double
plan of the same call."""
import numpy as np
import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

pytestmark = pytest.mark.gpu


def triangular(n, seed):
    """Triangular with a small diagonal: the permanent is the diagonal's product, the terms are far larger."""
    g = np.random.default_rng(seed)
    a = np.triu(synth.single_er(n, 0.3, seed, values="f64"), 1)
    a[np.arange(n), np.arange(n)] = g.uniform(0.15, 0.25, n)
    return np.ascontiguousarray(a[:, g.permutation(n)])


@pytest.mark.parametrize("n", [20, 24])
def test_auto_reruns_take_the_eliminated_walk(n):
    a = triangular(n, n)
    p = A.Plan(a)
    want, sa = oracle.nw_perm(a, threads=16)
    tol = 64 * n * (2.0 ** -104 + 2.0 ** -oracle.long_double_bits()) * float(sa)
    explicit = A.permanent(a, precision=A.PERM_PREC_DD)
    chained = A.permanent(a, precision=A.PERM_PREC_DD, ordering=A.PERM_ORDER_DEGREE)
    assert explicit.fp_ops_per_step < 0.5 * chained.fp_ops_per_step   # an eliminated walk
    for r in (p.compute(), p.compute(), A.permanent(a)):
        assert r.precision == A.PERM_PREC_DD
        assert abs((r.f64 - want.hi) + (r.f64_lo - want.lo)) <= tol
        assert r.fp_ops_per_step == explicit.fp_ops_per_step
    p.close()
