"""The device buffer and pinned memory of a plan go on to the next plan when it is
destroyed: nothing may be in flight on them by then, whatever its calls returned."""
import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

pytestmark = pytest.mark.gpu


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
