"""Plan creation of generated kernels: a build that was rejected (its step spills)
is remembered like one that was kept."""
import re

import pytest

from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,kw", [
    (lambda: synth.band_plus(48, 3, 2, seed=1, values="01"), {"g_hi": 1 << 30}),
    (lambda: synth.band_plus(48, 3, 2, seed=2, values="01"), {"g_hi": 1 << 30}),
    (lambda: synth.single_er(36, 0.2, 3, values="01", shuffle_cols=True), {}),
], ids=["band48_1", "band48_2", "er36"])
def test_a_second_plan_compiles_nothing(make, kw):
    a = A.CSRMatrix(make())
    src, k, _ = A.elim_source(a, **kw)
    widest = int(re.search(r"operations per outer step (\d+)", src).group(1)) / 2.0 ** k
    first = A.Plan(a, **kw)
    r = first.compute()
    if r.fp_ops_per_step < 1.01 * widest + 2.0 ** -k:
        pytest.skip("the widest build of this matrix is kept")
    try:
        A.inject_failures(A.PERM_SITE_NVRTC, 1)   # the next compilation fails
        second = A.Plan(a, **kw)
        s = second.compute()
        assert s.ms_compile == 0.0
        assert (s.value, s.partial_int, s.fp_ops_per_step) == (r.value, r.partial_int, r.fp_ops_per_step)
        with pytest.raises(A.PermError):          # it is still pending
            A.Plan(a, flags=A.PERM_FLAG_NO_KERNEL_CACHE, **kw)
    finally:
        A.inject_failures(A.PERM_SITE_NVRTC, 0)
    first.close()
    second.close()
