"""Sums of |terms| whose partial products leave FP32's range although the terms do
not: pairs of rows (1, -1 + d), (1, 1) on two columns of their own, so that every
term carries a factor d for each pair.  The eliminated walk multiplies magnitudes
in FP32 and is left to the chained walk there.  On the host, where it is planned,
its emulated sum is compared with the oracle's; on the GPU whatever runs is."""
import re

import numpy as np
import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth
from tests import test_elim_host_emulation as gen
from tests import test_vm_host_emulation as vm


def paired(n, pairs, d, seed, triangular=False):
    a = np.zeros((n, n))
    g = np.random.default_rng(seed)
    for i in range(0, 2 * pairs, 2):
        a[i, i:i + 2] = 1.0, -1.0 + d
        a[i + 1, i:i + 2] = 1.0, 1.0
    m = n - 2 * pairs
    rest = synth.single_er(m, 0.4, seed, values="f64")
    if triangular:   # the permanent is the diagonal's product, far below the sum of |terms|
        rest = np.triu(rest, 1) + np.diag(g.uniform(0.15, 0.25, m))
    a[2 * pairs:, 2 * pairs:] = rest
    a[2 * pairs:, :2 * pairs] = (g.random((m, 2 * pairs)) < 0.1) * g.random((m, 2 * pairs))
    return a


CASES = [(12, 1, -52), (16, 2, -40), (24, 4, -50), (26, 5, -45), (28, 3, -52), (28, 4, -52), (30, 4, -52)]


@pytest.mark.parametrize("n,pairs,d", CASES)
def test_planned_walks_have_the_sum_of_magnitudes(n, pairs, d):
    a = paired(n, pairs, 2.0 ** d, n)
    img, kind, k, order, scale, shift = A.elim_image(a)
    src, ks, orders = A.elim_source(a, flags=A.PERM_FLAG_ABS_SUM)
    found = [(k, order, shift, lambda K: vm.emulate(img, kind, K, [0])[0])] if img else []
    if src:
        found.append((ks, orders, int(re.search(r"int scale = (-?\d+);", src).group(1)), lambda K: gen.emulate(src, K, [0])[0]))
    for k, order, scale, run in found:
        h = n - 1 - k
        K = min(h, max(0, 16 - k))
        ao = np.ascontiguousarray(a[:, order[h:n - 1] + order[:h] + order[n - 1:]])
        _, sa = oracle.nw_range(ao, 0, 1 << (K + k))
        got = np.ldexp(np.array(run(K), dtype=np.uint64).view(np.float64)[2], scale)
        assert abs(got - float(sa)) <= 1e-4 * float(sa)


def test_ordinary_matrices_keep_the_eliminated_walk():
    """Values in (0,1], equal values, signed values, and rows 2^-200..2^200 apart."""
    g = np.random.default_rng(5)
    for n in (9, 17, 28, 36, 48):
        a = synth.single_er(n, 0.2, n, values="f64")
        for m in (a, (a != 0) * 0.3, a * g.choice([-1.0, 1.0], a.shape), a * np.exp2(np.linspace(-200, 200, n).round())[:, None]):
            assert A.elim_image(m)[0], n


@pytest.mark.gpu
@pytest.mark.parametrize("call", [A.permanent, A.permanent_noalloc, lambda a, **kw: A.batch([a], **kw)[0]],
                         ids=["plan", "noalloc", "batch"])
def test_sums_and_precision_on_the_gpu(call):
    for n, pairs, d in ((24, 4, -50), (28, 4, -52)):
        a = paired(n, pairs, 2.0 ** d, n)
        want, sa = oracle.nw_perm(a, threads=16)
        r = call(a)
        assert abs(r.value - float(want)) <= 1e-9 * abs(float(want))
        assert abs(r.abs_term_sum - float(sa)) <= 1e-4 * float(sa)
    a = paired(28, 4, 2.0 ** -52, 28, triangular=True)
    want, sa = oracle.nw_perm(a, threads=16)
    r = call(a)
    assert r.precision == A.PERM_PREC_DD   # n 2^-53 sum|terms| is far above 1e-9 |perm|
    assert abs(r.value - float(want)) <= 1e-9 * abs(float(want))
