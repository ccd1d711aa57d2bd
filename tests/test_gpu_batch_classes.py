"""perm_batch over matrices whose programs fall into every shared-memory class of
the eliminated walk, beside chained walks and double-double reruns: the same
bits through the graph and launched directly, one plan's values, the oracle's."""
import pytest

from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth
from tests.test_gpu_batch import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,n_lo,n_hi,p_lo,p_hi", [(24, 9, 16, 0.2, 0.45), (120, 12, 25, 0.1, 0.45)])
def test_every_class_in_one_batch(count, n_lo, n_hi, p_lo, p_hi):
    items = synth.batch(count, n_lo, n_hi, p_lo, p_hi, seed=77)
    mats = [A.CSRMatrix(it.a) for it in items]
    graph = A.batch(mats)
    direct = A.batch(mats, flags=A.PERM_FLAG_NO_GRAPH)
    alone = A.batch(mats, sequential=True)
    for it, g, d, s in zip(items, graph, direct, alone):
        assert g.status == d.status == s.status == 0
        assert g.value == d.value and g.abs_term_sum == d.abs_term_sum
        if it.values == "01":
            assert g.value == s.value
        else:   # n u sum|terms| each
            assert abs(g.value - s.value) <= 2 * it.a.shape[0] * 2.0 ** -53 * s.abs_term_sum
        if it.a.shape[0] <= 16:
            check(it, g)
