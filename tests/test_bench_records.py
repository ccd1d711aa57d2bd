"""What bench.py says about the kernel it times follows the library's sources."""
import os
import re

import bench
from paper_2501_15126_gb300 import _abi as A

CSRC = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_2501_15126_gb300", "csrc")


def test_the_kernel_hash_follows_the_kernel_that_runs(monkeypatch):
    """The n=36 workload runs the eliminated walk, so its source decides, not the chained walk's."""
    h = bench.kernel_hash()
    assert A.elim_source(bench.workload_matrix())[1] > 0
    source = A.elim_source
    monkeypatch.setattr(A, "elim_source", lambda a: (source(a)[0] + "// another",) + source(a)[1:])
    assert bench.kernel_hash() != h


def test_the_fused_task_limit_is_the_librarys():
    text = open(os.path.join(CSRC, "plan.hpp")).read()
    assert int(re.search(r"kFusedTasks = (\d+);", text).group(1)) == bench.FUSED_TASKS
