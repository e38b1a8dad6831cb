"""The native half of the Python binding: what it hands to the C-ABI, seen by a function of the same signature that records its
arguments (no GPU, no library call)."""
import ctypes as C

import pytest
import torch

import paper_2405_11095_b200 as F

NAMES = F._NATIVE_FUNCTIONS


@pytest.fixture
def calls():
    from paper_2405_11095_b200 import _native as n
    seen, keep = [], []
    for name in NAMES:
        argtypes = getattr(F.lib(), name).argtypes
        fn = C.CFUNCTYPE(C.c_int, *argtypes)(lambda *a, name=name: seen.append((name, a)) or -3)
        keep.append(fn)
    n.bind(tuple(C.cast(f, C.c_void_p).value for f in keep), lambda: 5, lambda dev: 1000 + dev, torch.float32, torch.bfloat16)
    yield n, seen
    F._calls = None      # the next call through the package binds the library again


@pytest.mark.parametrize("dtype,code", [(torch.float32, F.F32), (torch.bfloat16, F.BF16), (torch.float64, -1)])
@pytest.mark.parametrize("shape,stride,M,stride_out", [((24,), None, 1, 20), ((3, 24), None, 3, 24), ((3, 24), 16, 3, 16)])
def test_arguments_of_an_encode(calls, dtype, code, shape, stride, M, stride_out):
    n, seen = calls
    g, bits, ws = torch.zeros(shape, dtype=dtype), torch.zeros(8, dtype=torch.int32), torch.zeros(100, dtype=torch.uint8)
    assert n.encode(g, 20, bits, 0.5, 2**64 - 1, 7, 2**32 - 1, 10, ws, stride) == -3        # the function's own status
    name, a = seen.pop()
    assert name == "fosgd_encode"
    assert a == (g.data_ptr(), code, 20, stride_out, M, 2**32 - 1, 2**64 - 1, 7, 0.5, 10, bits.data_ptr(), ws.data_ptr(), 100, 1005)
    assert n.encode_measured_blocks(g, 20, bits, ws, None, 1, 2, 2.0, 3.0, 4, 10, None, ws, stride) == -3
    name, a = seen.pop()
    assert name == "fosgd_encode_measured_blocks"
    assert a == (g.data_ptr(), code, 20, stride_out, M, 4, 1, 2, 2.0, 3.0, 10, ws.data_ptr(), None, bits.data_ptr(), None, 0,
                 ws.data_ptr(), 100, 1005)


def test_errors_before_the_call(calls):
    n, seen = calls
    g, bits = torch.zeros(24), torch.zeros(8, dtype=torch.int32)
    with pytest.raises(TypeError):
        n.encode(g, 20, bits)                                            # too few arguments
    with pytest.raises(TypeError):
        n.encode(g, "20", bits, 0.5, 1, 2, 0, 0, None, None)             # not a number
    with pytest.raises(AttributeError):
        n.encode([1.0], 20, bits, 0.5, 1, 2, 0, 0, None, None)           # not a tensor
    with pytest.raises(TypeError):
        n.bind((0,) * len(NAMES), None, None, None)
    with pytest.raises(ValueError):
        n.bind((0,) * len(NAMES), None, None, None, None)
    assert not seen
