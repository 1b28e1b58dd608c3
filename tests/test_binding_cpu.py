"""The binding's handling of host buffers, without a GPU."""
import array
import ctypes

import numpy as np
import pytest

import paper_1701_04148_gb300 as sf


@pytest.mark.parametrize("buf", [bytearray(64), array.array("I", range(16)), memoryview(bytearray(64)),
                                 (ctypes.c_uint32 * 16)(), b"0123456789abcdef", [1, 2, 3]])
def test_only_arrays_and_tensors_have_host_addresses(buf):
    """A request's answers are four bytes each and their number is len(out): a bytearray of n bytes, taken for n
    answers, would be written past its end."""
    with pytest.raises(AttributeError):
        sf._host_ptr(buf)


def test_addresses_of_arrays():
    a = np.arange(12, dtype=np.uint32)
    ro = a.copy()
    ro.flags.writeable = False
    structured = np.zeros(4, np.dtype([("a", "<u4"), ("b", "<u2")]))
    times = np.zeros(3, "datetime64[s]")
    for x in (a, a[3:], a.reshape(3, 4), a[::2], ro, structured, times, a.view(np.recarray)):
        assert sf._host_ptr(x) == x.__array_interface__["data"][0]
    import torch
    t = torch.arange(5)
    assert sf._host_ptr(t) == t.data_ptr()
