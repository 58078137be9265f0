"""What the binding hands to the C ABI for buffers and streams (no GPU)."""
import ctypes

import numpy as np
import pytest

from paper_2004_02003_gb300 import bto


class _Buffer:
    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address


# Buffers are anything with a data_ptr() that int() takes, not torch tensors
# alone: ctypes itself would refuse a numpy integer.
@pytest.mark.parametrize("address", [0x7F0012345600, np.int64(0x7F0012345600), np.uint64(0x7F0012345600)])
def test_addresses_are_plain_integers(address):
    got = bto._addr(_Buffer(address))
    assert type(got) is int and got == 0x7F0012345600
    assert ctypes.c_void_p(got).value == got
    assert bto._addr(None) is None and bto._addr(5) == 5
