"""libmqgrad for B200: Python binding of the C ABI in include/mqgrad.h.

The binding only marshals arguments: torch CUDA tensors supply the device pointers and the
current torch stream supplies the CUDA stream; every step of the path runs in the CUDA
kernels of libmqgrad.so.  There is no CPU fallback: a missing library or a CPU tensor
raises.

Function names and argument order follow the C ABI:
  mqg_quantize, mqg_quantize_workers, mqg_dequant_accumulate, mqg_apply, mqg_server_step,
  mqg_server_requantize, mqg_quantize_segments, mqg_quantize_segments_workers, mqg_server_step_segments, mqg_quantize_minmax,
  mqg_quantize_workers_minmax,
  mqg_dequant_accumulate_minmax, mqg_server_step_minmax, mqg_quantize_l2, mqg_quantize_workers_l2, mqg_quantize_segments_l2,
  mqg_l2_workspace_floats, mqg_quantize_segments_l2_static, mqg_quantize_1bit_ef, mqg_code_words, mqg_num_buckets,
  mqg_wire_bytes, mqg_last_error, mqg_version, mqg_device_timeouts, mqg_check_timeouts,
  mqg_test_wait_override.
"""
from __future__ import annotations

import ctypes as C
import os

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libmqgrad.so")
_NOT_BUILT = "%s is not built (%s); run `python paper_1804_08066_b200/build.py`. There is no fallback path."

MQG_OK = 0
MQG_ERR_INVALID = -1
MQG_ERR_BITS = -2
MQG_ERR_ALIGN = -3
MQG_ERR_TOO_MANY_WORKERS = -4
MQG_ERR_CUDA = -5
MQG_ERR_TIMEOUT = -6
MQG_F32, MQG_BF16 = 0, 1
MQG_MAX_WORKERS = 32


class MqgError(RuntimeError):
    def __init__(self, status: int, message: str):
        super().__init__("libmqgrad status %d: %s" % (status, message))
        self.status = status


def _load() -> C.CDLL:
    if not os.path.exists(LIB_PATH):
        raise ImportError(_NOT_BUILT % ("libmqgrad.so", LIB_PATH))
    lib = C.CDLL(LIB_PATH)
    u64, u32, i32, vp, f32 = C.c_uint64, C.c_uint32, C.c_int, C.c_void_p, C.c_float
    sigs = {
        "mqg_code_words": (C.c_size_t, [u64, i32]),
        "mqg_num_buckets": (C.c_size_t, [u64, u64]),
        "mqg_wire_bytes": (C.c_size_t, [u64, i32, u64]),
        "mqg_last_error": (C.c_char_p, []),
        "mqg_version": (i32, []),
        "mqg_device_timeouts": (i32, [C.POINTER(C.c_uint)]),
        "mqg_check_timeouts": (i32, [C.POINTER(C.c_uint), i32]),
        "mqg_test_wait_override": (i32, [u32, i32]),
        "mqg_quantize": (i32, [vp, u64, i32, u64, u64, vp, vp, i32, u32, u32, u64, vp]),
        "mqg_quantize_workers": (i32, [vp, i32, u64, i32, u64, u64, vp, vp, i32, u32, u32, u64, vp]),
        "mqg_dequant_accumulate": (i32, [vp, vp, i32, i32, u64, vp, u64, i32, vp]),
        "mqg_apply": (i32, [vp, vp, f32, u64, vp]),
        "mqg_quantize_minmax": (i32, [vp, u64, i32, u64, vp, vp, i32, vp]),
        "mqg_quantize_workers_minmax": (i32, [vp, i32, u64, i32, u64, vp, vp, i32, vp]),
        "mqg_dequant_accumulate_minmax": (i32, [vp, vp, i32, i32, u64, vp, u64, i32, vp]),
        "mqg_server_step_minmax": (i32, [vp, vp, i32, i32, u64, u64, vp, f32, vp, vp]),
        "mqg_server_step": (i32, [vp, vp, i32, i32, u64, u64, vp, f32, vp, vp]),
        "mqg_server_requantize": (i32, [vp, vp, i32, i32, u64, u64, f32, u64, vp, vp, u32, u32, vp]),
        "mqg_quantize_segments": (i32, [vp, i32, vp, vp, i32, u64, vp, vp, i32, u32, u32, u64, vp]),
        "mqg_server_step_segments": (i32, [vp, vp, i32, i32, i32, vp, vp, vp, f32, vp, vp]),
        "mqg_quantize_segments_workers": (i32, [vp, i32, i32, vp, vp, i32, u64, vp, vp, i32, u32, u32, u64, vp]),
        "mqg_quantize_1bit_ef": (i32, [vp, vp, u64, u64, vp, vp, i32, vp]),
        "mqg_quantize_l2": (i32, [vp, u64, i32, u64, u64, vp, vp, i32, u32, u32, u64, vp]),
        "mqg_quantize_workers_l2": (i32, [vp, i32, u64, i32, u64, u64, vp, vp, i32, u32, u32, u64, vp]),
        "mqg_l2_workspace_floats": (C.c_size_t, [i32, vp]),
        "mqg_quantize_segments_l2": (i32, [vp, i32, vp, vp, i32, u64, vp, vp, i32, u32, u32, u64, vp,
                                           C.c_size_t, vp]),
        "mqg_quantize_segments_l2_static": (i32, [vp, i32, vp, vp, i32, u64, vp, vp, i32, u32, u32, u64, vp]),
    }
    for name, (res, args) in sigs.items():
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    return lib


class _LazyLibrary:
    """Loads libmqgrad.so at the first call instead of at import, so that a process which only
    imports the input generators (workloads.py) never maps the library."""

    def __init__(self):
        self._lib = None

    def __getattr__(self, name):
        if self._lib is None:
            self._lib = _load()
        return getattr(self._lib, name)


_lib = _LazyLibrary()


def _check(status: int) -> None:
    if status != MQG_OK:
        raise MqgError(status, _lib.mqg_last_error().decode())


def _u64_table(values):
    vals = [int(v) for v in values]
    return (C.c_uint64 * len(vals))(*vals)


# The calls that enqueue work are native functions (csrc/mqg_binding.cpp; its file: build.binding_path): the device is
# done with a small gradient in less time than Python and ctypes need to marshal a call's arguments.
_NATIVE = frozenset((
    "mqg_quantize", "mqg_quantize_workers", "mqg_dequant_accumulate", "mqg_apply", "mqg_server_step",
    "mqg_server_requantize", "mqg_quantize_segments", "mqg_quantize_segments_workers", "mqg_server_step_segments",
    "mqg_quantize_minmax", "mqg_quantize_workers_minmax", "mqg_dequant_accumulate_minmax", "mqg_server_step_minmax",
    "mqg_quantize_l2", "mqg_quantize_workers_l2", "mqg_quantize_segments_l2", "mqg_quantize_segments_l2_static",
    "mqg_quantize_1bit_ef"))


def _native(name):
    """The native function `name`; the first call loads them all."""
    if name not in globals():
        import importlib.util

        from .build import binding_path
        path = binding_path()              # imports torch: its libraries have to be loaded before the native module's
        for file in (LIB_PATH, path):
            if not os.path.exists(file):
                raise ImportError(_NOT_BUILT % (os.path.basename(file), file))
        spec = importlib.util.spec_from_file_location(__name__ + "._binding", path)
        native = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(native)
        native._set_error_class(MqgError)
        for fn in _NATIVE:
            getattr(native, fn).__module__ = __name__      # found here when a pickle names it
            globals()[fn] = getattr(native, fn)
    return globals()[name]


def __getattr__(name):
    """Loads the native functions when the first of them is asked for, not at import (as _LazyLibrary)."""
    if name not in _NATIVE:
        raise AttributeError("module %r has no attribute %r" % (__name__, name))
    try:
        return _native(name)
    except ImportError:
        def not_built(*args, **kwargs):                    # the name is there all the same; a call says what is missing
            return _native(name)(*args, **kwargs)
        not_built.__name__ = not_built.__qualname__ = name
        return not_built


def __dir__():
    return sorted({*globals(), *_NATIVE})


def mqg_code_words(n: int, bits: int) -> int:
    return int(_lib.mqg_code_words(n, bits))


def mqg_num_buckets(n: int, bucket: int) -> int:
    return int(_lib.mqg_num_buckets(n, bucket))


def mqg_wire_bytes(n: int, bits: int, bucket: int) -> int:
    return int(_lib.mqg_wire_bytes(n, bits, bucket))


def mqg_last_error() -> str:
    return _lib.mqg_last_error().decode()


def mqg_version() -> int:
    return int(_lib.mqg_version())


def mqg_device_timeouts() -> int:
    """Number of kernel waits that gave up on the current device (synchronises); 0 when healthy."""
    c = C.c_uint(0)
    _check(_lib.mqg_device_timeouts(C.byref(c)))
    return int(c.value)


def mqg_check_timeouts(reset: bool = True) -> int:
    """Waits that ran out on the current device since the last reset (synchronises).  Raises MqgError
    with status MQG_ERR_TIMEOUT when there were any, after clearing the counter if `reset`; returns 0
    otherwise."""
    c = C.c_uint(0)
    _check(_lib.mqg_check_timeouts(C.byref(c), 1 if reset else 0))
    return int(c.value)


def mqg_test_wait_override(poll_limit: int = 0, arm_only: bool = False) -> None:
    """Test hook of the C ABI (see include/mqgrad.h); (0, False) restores normal operation."""
    _check(_lib.mqg_test_wait_override(poll_limit, 1 if arm_only else 0))


def mqg_l2_workspace_floats(seg_off) -> int:
    return int(_lib.mqg_l2_workspace_floats(len(seg_off) - 1, _u64_table(seg_off)))


MQG_L2_STATIC_WORKSPACE_FLOATS = 65536


def raw_library() -> C.CDLL:
    """The ctypes handle, for callers that pass raw device pointers themselves."""
    _lib.mqg_version                       # loads the library if this is its first use
    return _lib._lib


__all__ = [_name for _name in __dir__() if not _name.startswith("_")]     # the native functions among them
