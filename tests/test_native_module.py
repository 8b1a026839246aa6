"""The native module's conversions and error handling, on the CPU: what the ctypes binding accepted and raised."""
import numpy as np
import pytest
import torch
from torch.utils._python_dispatch import TorchDispatchMode

from paper_2503_18893_b200 import xkv


class _Refuse(TorchDispatchMode):
    def __init__(self, error):
        super().__init__()
        self.error = error

    def __torch_dispatch__(self, func, types, args=(), kwargs=None):
        raise self.error


@pytest.mark.parametrize("error", [KeyError("no memory of that kind"), torch.OutOfMemoryError("out of memory"), MemoryError()])
def test_an_error_of_the_allocation_keeps_its_type(error):
    x = torch.zeros((4, 64), dtype=torch.bfloat16)
    codes, meta = torch.zeros((4, 32), dtype=torch.uint8), torch.zeros((4, 2), dtype=torch.int32)
    for call in (lambda: xkv._xkv.quantize_rtn(x, 4, 0), lambda: xkv._xkv.dequantize_rtn(codes, meta, 4, 0)):
        with _Refuse(error), pytest.raises(type(error)):
            call()


@pytest.mark.parametrize("stream", [0, np.int64(0), np.uint64(0), True])
def test_streams_that_convert_to_an_integer(stream):
    # no handle: the call is refused by the library, after its arguments have been converted
    assert xkv._xkv.sr_select(0, 0, 1, None, 8, None, None, stream) == xkv.XKV_ERR_INVALID_ARG


@pytest.mark.parametrize("stream", ["0x10", object(), 1.5j])
def test_streams_that_are_none(stream):
    with pytest.raises((TypeError, ValueError)):
        xkv._xkv.sr_select(0, 0, 1, None, 8, None, None, stream)
