"""The host's record of a resident kernel's counters follows the launches that were made."""
import pytest
import torch

from tests import internals

pytestmark = pytest.mark.skipif(torch.cuda.is_available(), reason="needs launches that fail: no device")


@pytest.fixture(scope="module")
def lib():
    return internals.load()


def test_sliced_kernel(lib):
    """A launch that fails counts nothing on the device, and the next one must not wait for it."""
    base = internals.uints(74, 19, 0)
    some = internals.pointers(*[256] * 16)
    assert lib.t_slices(256, 512, 60, 3, 148, some, base, None) != 0
    assert list(base) == [74, 19, 0]


def test_batch_kernel(lib):
    base = internals.uints(74, 592, 19)
    assert lib.t_batch_record(base) != 0
    assert list(base) == [74, 592, 19]
