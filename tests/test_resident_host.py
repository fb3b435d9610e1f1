"""Host side of the resident kernels: the record of their counters, the shapes they take."""
import pytest
import torch

from tests import internals

no_device = pytest.mark.skipif(torch.cuda.is_available(), reason="needs launches that fail: no device")


@pytest.fixture(scope="module")
def lib():
    return internals.load()


@no_device
def test_record_of_the_sliced_kernel(lib):
    """A launch that fails counts nothing on the device, and the next one must not wait for it."""
    base = internals.uints(74, 19, 0)
    some = internals.pointers(*[256] * 16)
    assert lib.t_slices(256, 512, 60, 3, 148, some, base, None) != 0
    assert list(base) == [74, 19, 0]


@no_device
def test_record_of_the_batch_kernel(lib):
    base = internals.uints(74, 592, 19)
    assert lib.t_batch_record(base) != 0
    assert list(base) == [74, 592, 19]


@pytest.mark.parametrize("sms", [100, 144, 148])
def test_widths_of_the_sliced_kernel(lib, sms):
    """Every multiple of 16 from 64 to 8192 at every capacity the library takes: its ring always has room."""
    for D in range(64, 8193, 16):
        for C in (1, 37, 512, 2752, 11008, 20480, 40960):
            for k in {1, C // 4 + 1, C}:
                assert lib.t_slices_supported(D, C, k, sms), (D, C, k)
    assert not lib.t_slices_supported(48, 512, 60, sms) and not lib.t_slices_supported(8208, 512, 60, sms)
