"""The device buffer and pinned memory of a plan go on to the next plan when it is
destroyed: nothing may be in flight on them by then, whatever its calls returned."""
import os
import subprocess
import sys

import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("kw", [{"engine": A.PERM_ENGINE_GENERIC}, {"engine": A.PERM_ENGINE_GENERIC, "chunk_log2": 5},
                                {"engine": A.PERM_ENGINE_CODEGEN}], ids=["table_program", "chained", "generated"])
def test_a_failed_compute_returns_with_its_stream_idle(kw):
    """The walk's launch fails (injected) after the upload was queued behind other
    work: the call waits for it, and the next plan, on another stream, is right."""
    import torch
    a, b = synth.single_er(16, 0.3, 61, values="01"), synth.single_er(17, 0.3, 62, values="01")
    busy, other = torch.cuda.Stream(), torch.cuda.Stream()
    try:
        p = A.Plan(a, **kw)
        with torch.cuda.stream(busy):
            torch.cuda._sleep(200_000_000)   # about 0.1 s
        A.inject_failures(A.PERM_SITE_LAUNCH, 1)
        with pytest.raises(A.PermError) as e:
            p.compute(busy.cuda_stream)
        assert e.value.status == A.PERM_ERR_CUDA
        assert busy.query()
        p.close()
        q = A.Plan(b, **kw)
        for _ in range(2):
            assert q.compute(other.cuda_stream).value == oracle.ryser_gray(b)
        q.close()
    finally:
        A.inject_failures(A.PERM_SITE_LAUNCH, 0)


RESET = """
import ctypes, sys
from paper_2501_15126_gb300 import _abi as A, synth
a, b = synth.single_er(14, 0.3, 1, values="01"), synth.single_er(15, 0.3, 2, values="f64")
def both(**kw):
    return [A.permanent(m, engine=A.PERM_ENGINE_GENERIC, **kw).value for m in (a, b)]
want = both() + both(chunk_log2=5)
kept = [A.Plan(m, engine=A.PERM_ENGINE_GENERIC) for m in (a, b, a, b)]
for p in kept:
    p.compute()
    p.close()
assert ctypes.CDLL("libcudart.so.13").cudaDeviceReset() == 0
plans = [A.Plan(m, engine=A.PERM_ENGINE_GENERIC) for m in (a, b, a, b)]
assert [p.compute().value for p in plans] == want[:2] * 2
assert both() + both(chunk_log2=5) == want
"""


def test_plans_after_a_device_reset_take_buffers_of_the_new_context():
    """cudaDeviceReset ends the process's own context and frees what it held; a plan
    created afterwards gets none of it.  In a process of its own."""
    subprocess.run([sys.executable, "-c", RESET], cwd=ROOT, check=True, timeout=300)


CONTEXTS = """
import ctypes
from paper_2501_15126_gb300 import _abi as A, synth
cu = ctypes.CDLL("libcuda.so.1")
a, b = synth.single_er(14, 0.3, 1, values="01"), synth.single_er(15, 0.3, 2, values="f64")
def both():
    return [A.permanent(m, engine=A.PERM_ENGINE_GENERIC).value for m in (a, b)]
want = both()
ctx, old = ctypes.c_void_p(), ctypes.c_void_p()
assert cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, 0) == 0       # current from here on
assert both() == want
assert cu.cuCtxPopCurrent_v2(ctypes.byref(old)) == 0
assert both() == want
assert cu.cuCtxPushCurrent_v2(ctx) == 0
assert both() == want and both() == want
assert cu.cuCtxPopCurrent_v2(ctypes.byref(old)) == 0
"""


def test_plans_in_a_context_of_the_callers_own_take_its_buffers():
    """A driver context beside the device's primary one, by turns."""
    subprocess.run([sys.executable, "-c", CONTEXTS], cwd=ROOT, check=True, timeout=300)
