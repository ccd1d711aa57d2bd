"""GPU test of the final reduction over task results: one block up to 512
tasks, several beyond, with a ragged last block.  Sub-ranges of exactly `tasks`
32-chunk tasks of 2^5 steps (the generic walk at an explicit chunk length)
against the oracle: exact bit for bit, FP64 within 64 n 2^-53 sum|terms|."""
import numpy as np
import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tasks", [1, 31, 128, 511, 512, 513, 1024, 1537, 4095])
def test_sums_over_any_number_of_tasks(tasks):
    n = 24
    for values in ("01", "f64"):
        a = synth.single_er(n, 0.3, 77, values=values)
        ao = np.ascontiguousarray(a[:, list(A.inspect(a).col_order)[:n]])
        hi = tasks << 10
        r = A.permanent(a, engine=A.PERM_ENGINE_GENERIC, chunk_log2=5, g_hi=hi)
        if values == "01":
            mask = (1 << (64 * min(r.exact_words, 2))) - 1
            assert r.partial_int & mask == oracle.nw2_range(ao, 0, hi, threads=16) & mask
        else:
            s, sa = oracle.nw_range(ao, 0, hi, threads=16)
            assert abs((r.f64 - s.hi) + (r.f64_lo - s.lo)) <= 64 * n * 2.0 ** -53 * float(sa)
            assert abs(r.abs_term_sum - float(sa)) <= 1e-4 * float(sa)
            assert abs(r.f64_lo) <= 2.0 ** -52 * abs(r.f64)   # the pair comes back normalised
