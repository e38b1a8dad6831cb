"""csrc/binding.c in Python and ctypes, for interpreters without headers to build it against: the same functions, 3 us a call
instead of 1."""
import ctypes as C

F32, BF16 = 0, 1
_fn, _get_device, _get_stream, _dtypes = (), None, None, {}


def bind(addresses, get_device, get_stream, float32, bfloat16):
    global _fn, _get_device, _get_stream, _dtypes
    from . import _NATIVE_FUNCTIONS, lib
    _fn = {name: C.CFUNCTYPE(C.c_int, *getattr(lib(), name).argtypes)(address)
           for name, address in zip(_NATIVE_FUNCTIONS, addresses, strict=True)}
    _get_device, _get_stream, _dtypes = get_device, get_stream, {float32: F32, bfloat16: BF16}


def _ptr(t):
    return 0 if t is None else t.data_ptr()


def _scratch(t):
    return _ptr(t), 0 if t is None else t.numel() * t.element_size()


def _rows(t):
    return t.size(0) if t.dim() == 2 else 1


def _grads(t, d, stride):
    """pointer, type, d, row stride, rows"""
    if stride is None:
        stride = t.stride(0) if t.dim() == 2 else d
    return t.data_ptr(), _dtypes.get(t.dtype, -1), d, stride, _rows(t)


def _amplitude(lam):
    """value, device pointer"""
    return (float(lam), 0) if isinstance(lam, (int, float)) else (0.0, _ptr(lam))


def _call(name, *args):
    return _fn[name](*args, _get_stream(_get_device()))


def encode(grads, d, bits, lam, seed, step, id0, b, ws, stride):
    return _call("fosgd_encode", *_grads(grads, d, stride), id0, seed, step, lam, b, _ptr(bits), *_scratch(ws))


def flatten(grads, d, out, seed, step, id0, b, ws, stride):
    return _call("fosgd_flatten", *_grads(grads, d, stride), id0, seed, step, b, _ptr(out), *_scratch(ws))


def decode(bits, d, out, lam, seed, step, worker_id, b, ws):
    return _call("fosgd_decode", _ptr(bits), d, worker_id, seed, step, lam, b, _ptr(out), *_scratch(ws))


def server_aggregate(bits, d, acc, lam, seed, step, total, id0, flags, lam_s, K, down, b, ws):
    M = _rows(bits)
    return _call("fosgd_server_aggregate", _ptr(bits), d, M, id0, M if total is None else total, seed, step, lam, b, _ptr(acc),
                 flags, lam_s, K, _ptr(down), *_scratch(ws))


def server_aggregate_dev(bits, d, acc, lam, seed, step, total, id0, flags, lam_s, K, down, b, per_block, ws):
    M = _rows(bits)
    return _call("fosgd_server_aggregate_dev", _ptr(bits), d, M, id0, M if total is None else total, seed, step, _ptr(lam),
                 _ptr(lam_s), int(per_block), b, _ptr(acc), flags, K, _ptr(down), *_scratch(ws))


def downlink_decode(down, d, out, lam_s, seed, step, K, b, ws):
    return _call("fosgd_downlink_decode", _ptr(down), d, seed, step, lam_s, K, b, _ptr(out), *_scratch(ws))


def downlink_decode_dev(down, d, out, lam_s, seed, step, K, b, per_block, ws):
    return _call("fosgd_downlink_decode_dev", _ptr(down), d, seed, step, _ptr(lam_s), int(per_block), K, b, _ptr(out),
                 *_scratch(ws))


def downlink_encode(gbar, d, down, lam_s, seed, step, K, b, per_block, ws):
    return _call("fosgd_downlink_encode", _ptr(gbar), d, seed, step, *_amplitude(lam_s), int(per_block), K, b, _ptr(down),
                 *_scratch(ws))


def downlink_apply(down, d, x, lam_s, seed, step, step_size, K, b, per_block, ws):
    return _call("fosgd_downlink_apply", _ptr(down), d, seed, step, *_amplitude(lam_s), int(per_block), K, b, float(step_size),
                 _ptr(x), *_scratch(ws))


def amplitudes(grads, d, lam, lam_s, alpha, alpha_s, b, per_block, ws, stride):
    return _call("fosgd_amplitudes", *_grads(grads, d, stride), alpha, alpha_s, b, int(per_block), _ptr(lam), _ptr(lam_s),
                 *_scratch(ws))


def encode_dev(grads, d, bits, lam, seed, step, id0, b, per_block, ws, stride):
    return _call("fosgd_encode_dev", *_grads(grads, d, stride), id0, seed, step, _ptr(lam), int(per_block), b, _ptr(bits),
                 *_scratch(ws))


def _measured(name, grads, d, bits, lam, lam_s, seed, step, alpha, alpha_s, id0, b, ws, amp_ws, stride):
    return _call(name, *_grads(grads, d, stride), id0, seed, step, alpha, alpha_s, b, _ptr(lam), _ptr(lam_s), _ptr(bits),
                 *_scratch(ws), *_scratch(amp_ws))


def encode_measured(*args):
    return _measured("fosgd_encode_measured", *args)


def encode_measured_blocks(*args):
    return _measured("fosgd_encode_measured_blocks", *args)
