"""The native half of the Python binding: whose build it is, and what takes its place where it cannot be built (no GPU)."""
import ctypes as C
import importlib.util
import inspect
import os
import sysconfig

import pytest
import torch

import paper_2405_11095_b200 as F


def build_module():
    spec = importlib.util.spec_from_file_location("fosgd_build", os.path.join(os.path.dirname(F.__file__), "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_the_extension_is_this_interpreters():
    from paper_2405_11095_b200 import _native
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert suffix != ".so" and _native.__file__.endswith("_native" + suffix)
    assert not os.path.exists(os.path.join(os.path.dirname(F.__file__), "_native.so"))


def test_a_build_without_headers_goes_on(monkeypatch, tmp_path):
    b = build_module()
    monkeypatch.setattr(b, "NATIVE_SO", str(tmp_path / "_native.so"))
    monkeypatch.setattr(b.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    assert b.build_binding(force=True) is None and not os.listdir(tmp_path)


def arguments(module, name, grads):
    """One call of every kind, with an argument of its own in every place; bits: a matrix of as many rows as the gradients."""
    t = [torch.zeros(k + 8, dtype=torch.int32) for k in range(8)]
    bits = torch.zeros(3, 8, dtype=torch.int32) if grads.dim() == 2 else t[0]
    return {
        "encode": (grads, 20, t[1], 0.5, 2**64 - 1, 7, 2**32 - 1, 10, t[2], None),
        "flatten": (grads, 20, t[1], 3, 7, 4, 10, None, 24),
        "decode": (t[1], 20, t[2], 0.5, 3, 7, 4, 10, t[3]),
        "server_aggregate": (bits, 20, t[1], 0.5, 3, 7, None, 4, 3, 0.25, 15, t[2], 10, t[3]),
        "server_aggregate_dev": (bits, 20, t[1], t[2], 3, 7, 9, 4, 1, t[3], 15, None, 10, True, t[4]),
        "downlink_decode": (t[1], 20, t[2], 0.5, 3, 7, 15, 10, t[3]),
        "downlink_decode_dev": (t[1], 20, t[2], t[3], 3, 7, 15, 10, 1, None),
        "downlink_encode": (t[1], 20, t[2], 0.5, 3, 7, 15, 10, False, t[3]),
        "downlink_apply": (t[1], 20, t[2], t[3], 3, 7, 0.125, 15, 10, True, t[4]),
        "amplitudes": (grads, 20, t[1], None, 2.0, 3.0, 10, False, t[2], 24),
        "encode_dev": (grads, 20, t[1], t[2], 3, 7, 4, 10, True, t[3], None),
        "encode_measured": (grads, 20, t[1], t[2], t[3], 3, 7, 2.0, 3.0, 4, 10, t[4], t[5], None),
        "encode_measured_blocks": (grads, 20, t[1], t[2], None, 3, 7, 2.0, 3.0, 4, 10, None, t[5], 24),
    }[name], t


@pytest.mark.parametrize("shape,dtype", [((24,), torch.float32), ((3, 24), torch.bfloat16), ((3, 24), torch.float64)])
def test_ctypes_hands_over_the_same_arguments(shape, dtype):
    from paper_2405_11095_b200 import _marshal, _native
    seen, keep = [], []
    for name in F._NATIVE_FUNCTIONS:
        keep.append(C.CFUNCTYPE(C.c_int, *getattr(F.lib(), name).argtypes)(lambda *a, name=name: seen.append((name, a)) or -3))
    addresses = tuple(C.cast(f, C.c_void_p).value for f in keep)
    grads = torch.zeros(shape, dtype=dtype)
    try:
        for m in (_marshal, _native):
            m.bind(addresses, lambda: 5, lambda dev: 1000 + dev, torch.float32, torch.bfloat16)
        for fn in F._NATIVE_FUNCTIONS:
            name = fn.removeprefix("fosgd_")
            args, _keep = arguments(F, name, grads)
            assert getattr(_marshal, name)(*args) == getattr(_native, name)(*args) == -3
            (a, mine), (b, theirs) = seen[-2:]
            assert a == b == fn and mine == theirs, name
    finally:
        F._calls = None      # the next call through the package binds the library again
    assert len(seen) == 2 * len(F._NATIVE_FUNCTIONS)
    assert all(inspect.isfunction(getattr(_marshal, fn.removeprefix("fosgd_"))) for fn in F._NATIVE_FUNCTIONS)
