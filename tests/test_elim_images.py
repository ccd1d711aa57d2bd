"""Every matrix that the host emulation of program images lists has an image: a case
without one is skipped there."""
import pytest

from paper_2501_15126_gb300 import _abi as A
from tests.test_vm_host_emulation import CASES


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("name,make,kw", CASES, ids=[c[0] for c in CASES])
def test_the_listed_matrices_have_images(name, make, kw, shared):
    assert A.elim_image(make(), shared_launch=shared, **kw)[0]
