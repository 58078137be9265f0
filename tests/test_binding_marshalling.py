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


class _Stream:
    cuda_stream = 0x5500


# Without a stream the call goes on torch's current one, asked for by its raw
# handle where torch has the calls, and through its public object where it has
# not (or before torch has a CUDA context).
@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice", None])
@pytest.mark.parametrize("initialised", [True, False])
def test_current_stream_with_and_without_the_raw_handle(monkeypatch, missing, initialised):
    import torch
    monkeypatch.setattr(bto, "_current", None, raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: initialised)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: _Stream)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 0x7700 + d, raising=False)
    if missing:
        monkeypatch.delattr(torch._C, missing)
    for _ in range(2):
        assert bto._stream(None) == (0x7703 if initialised and not missing else 0x5500)
    assert bto._stream(9) == 9 and bto._stream(_Stream) == 0x5500
