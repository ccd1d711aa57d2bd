"""perm_batch with long walks: the memory for their task results."""
import pytest

from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

pytestmark = pytest.mark.gpu


def test_long_chained_walks_fit_one_batch():
    """24 dense matrices of n = 44 with a deadline, which keeps the chained walk: 2^26
    tasks and 1.6 GB each at 2^12 steps a chunk (8 times that would not fit the GPU).
    The deadline stops them."""
    mats = [synth.single_er(44, 0.5, s, values="f64") for s in range(24)]
    assert [r.status for r in A.batch(mats, timeout_ms=20)] == [A.PERM_ERR_TIMEOUT] * 24
