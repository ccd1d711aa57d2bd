"""The allocation-free call on threads of small stacks: what its planner needs is not
on the stack (some 60 KB are)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CALLS = """
import threading
from paper_2501_15126_gb300 import _abi as A, synth
mats = [A.CSRMatrix(synth.single_er(n, 0.3, n, values=v)) for n in (12, 24) for v in ("01", "f64")]
want = [A.permanent_noalloc(m).value for m in mats]
got = []
def calls():
    for m in mats:
        got.append(A.permanent_noalloc(m).value)
        A.permanent_noalloc(m, precision=A.PERM_PREC_DD)
threading.stack_size(160 * 1024)
for _ in range(2):
    t = threading.Thread(target=calls)
    t.start()
    t.join()
assert got == want * 2, (got, want)
"""


def test_noalloc_on_a_thread_of_160_kb():
    """In a process of its own: an overflow ends the process."""
    subprocess.run([sys.executable, "-c", CALLS], cwd=ROOT, check=True, timeout=300)
