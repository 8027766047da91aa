"""Binding of libogq.so: same names and argument order as include/ogq.h.

The data-path calls are functions of the C module `_native` (argument conversion in ctypes took longer than
many of the kernels); the host-only helpers and the measurement helpers go through ctypes.
"""
from __future__ import annotations

import ctypes
import os
from typing import Optional, Sequence

import numpy as np

_HERE = os.path.dirname(os.path.abspath(__file__))
_LIB_PATH = os.path.join(_HERE, "libogq.so")

OGQ_BINGRAD_PB, OGQ_BINGRAD_B, OGQ_ORQ = 0, 1, 2
OGQ_ST_EMPTY, OGQ_ST_NONFINITE, OGQ_ST_CONSTANT, OGQ_ST_ITER_CAP, OGQ_ST_INTERNAL = 1, 2, 4, 8, 16

_STATUS_NAMES = {1: "OGQ_ERR_INVALID_ARG", 2: "OGQ_ERR_UNSUPPORTED", 3: "OGQ_ERR_WORKSPACE", 4: "OGQ_ERR_CUDA",
                 5: "OGQ_ERR_LIMIT"}


class OgqError(RuntimeError):
    def __init__(self, code: int, where: str):
        super().__init__(f"{where} failed: {_STATUS_NAMES.get(code, code)}")
        self.code = code


_lib: Optional[ctypes.CDLL] = None


def lib_path() -> str:
    return _LIB_PATH


def lib() -> ctypes.CDLL:
    """The loaded library.  Raises if libogq.so has not been built (no fallback exists)."""
    global _lib
    if _lib is None:
        if not os.path.exists(_LIB_PATH):
            raise ImportError(
                f"{_LIB_PATH} is missing: build it with `python -m paper_2002_11082_b200.build` "
                "(nvcc, sm_100a); there is no CPU fallback"
            )
        L = ctypes.CDLL(_LIB_PATH)
        vp, i64, i32, sz = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_size_t
        L.ogq_version.restype = ctypes.c_char_p
        L.ogq_version.argtypes = []
        L.ogq_bits_for_levels.restype = i32
        L.ogq_bits_for_levels.argtypes = [i32]
        L.ogq_packed_layout.restype = i32
        L.ogq_packed_layout.argtypes = [vp, i32, i32, vp]
        L.ogq_workspace_bytes.restype = sz
        L.ogq_workspace_bytes.argtypes = [i32, i64, i32]
        L.ogq_bucket_packed_words.restype = i64
        L.ogq_bucket_packed_words.argtypes = [i64, i32, i32]
        L.ogq_dense_digits.restype = i32
        L.ogq_dense_digits.argtypes = [i32]
        L.ogq_dense_layout.restype = i32
        L.ogq_dense_layout.argtypes = [vp, i32, i32, vp]
        L.ogq_launch_count.restype = ctypes.c_ulonglong
        L.ogq_launch_count.argtypes = []
        L.ogq_profile_enable.restype = i32
        L.ogq_profile_enable.argtypes = [i32]
        L.ogq_profile_collect.restype = i32
        L.ogq_profile_collect.argtypes = [vp, vp, i32, i32]
        _lib = L
    return _lib


def _check(code: int, where: str) -> None:
    if code != 0:
        raise OgqError(code, where)


_DATA_PATH = (
    "ogq_levels_bingrad", "ogq_levels_bingrad_b_noalloc", "ogq_levels_orq", "ogq_quantize_pack", "ogq_unpack_sum",
    "ogq_clip_threshold", "ogq_levels_orq_clipped", "ogq_levels_bingrad_clipped", "ogq_quant_error",
    "ogq_expected_error", "ogq_quantize_pack_dense", "ogq_unpack_sum_dense", "ogq_quantize_pack_clipped",
    "ogq_bucket_encode", "ogq_bucket_decode_sum",
)


def _attach() -> None:
    """Gives the C module the addresses of the library's functions (before its first call)."""
    L = lib()
    _native_module().set_addresses({n: ctypes.cast(getattr(L, n), ctypes.c_void_p).value for n in _DATA_PATH})


def _first_device() -> int:
    """The current device, for the first call without a stream: brings torch's CUDA state up, after which the
    C module asks torch directly."""
    import torch

    torch.cuda.current_stream()
    _native_module().setup(_attach, _check, torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream)
    return torch._C._cuda_getDevice()


def _first_raw_stream(device: int) -> int:
    import torch

    return torch._C._cuda_getCurrentRawStream(device)


def _native_module():
    try:
        from . import _native
    except ImportError as e:
        raise ImportError(
            "the C module of the binding is missing: build it with `python -m paper_2002_11082_b200.build`; "
            "there is no other path to the library's data-path calls"
        ) from e
    return _native


def _entry(name: str):
    try:
        return getattr(_native_module(), name)
    except ImportError:
        # imported before the build: looked up again at every call
        def late(*args, **kwargs):
            _setup_native()
            return getattr(_native_module(), name)(*args, **kwargs)

        late.__name__ = name
        return late


def _setup_native() -> None:
    _native_module().setup(_attach, _check, _first_device, _first_raw_stream)


try:
    _setup_native()
except ImportError:
    pass

for _name in _DATA_PATH:
    globals()[_name] = _entry(_name)


def ogq_version() -> str:
    return lib().ogq_version().decode()


def ogq_bits_for_levels(s: int) -> int:
    return int(lib().ogq_bits_for_levels(int(s)))


def ogq_packed_layout(h_off, bits: int) -> np.ndarray:
    """Host helper: word offsets [T+1] of the packed regions for element offsets h_off [T+1]."""
    h = np.ascontiguousarray(np.asarray(h_off), dtype=np.int64)
    out = np.zeros_like(h)
    _check(lib().ogq_packed_layout(h.ctypes.data, h.size - 1, int(bits), out.ctypes.data), "ogq_packed_layout")
    return out


def ogq_workspace_bytes(num_tensors: int, total_elems: int, max_levels: int) -> int:
    return int(lib().ogq_workspace_bytes(int(num_tensors), int(total_elems), int(max_levels)))


def ogq_bucket_packed_words(total_elems: int, d: int, bits: int) -> int:
    return int(lib().ogq_bucket_packed_words(int(total_elems), int(d), int(bits)))


def ogq_dense_digits(s: int) -> int:
    return int(lib().ogq_dense_digits(int(s)))


def ogq_dense_layout(h_off, s: int) -> np.ndarray:
    """Host helper: word offsets [T+1] of the base-s packed regions for element offsets h_off [T+1]."""
    h = np.ascontiguousarray(np.asarray(h_off), dtype=np.int64)
    out = np.zeros_like(h)
    _check(lib().ogq_dense_layout(h.ctypes.data, h.size - 1, int(s), out.ctypes.data), "ogq_dense_layout")
    return out


def ogq_launch_count() -> int:
    return int(lib().ogq_launch_count())


def ogq_profile_enable(on: bool) -> None:
    lib().ogq_profile_enable(1 if on else 0)


def ogq_profile_collect(max_records: int = 65536):
    """Returns [(kernel name, milliseconds), ...] for the launches recorded since profiling was enabled."""
    ms = np.zeros(max_records, dtype=np.float32)
    stride = 48
    names = ctypes.create_string_buffer(max_records * stride)
    n = lib().ogq_profile_collect(ms.ctypes.data, ctypes.cast(names, ctypes.c_void_p), stride, max_records)
    raw = names.raw
    return [(raw[i * stride : (i + 1) * stride].split(b"\0", 1)[0].decode(), float(ms[i])) for i in range(n)]


def device_pointer_array(tensors: Sequence, device=None):
    """An int64 device tensor holding the data pointers of `tensors` (for ogq_unpack_sum)."""
    import torch

    dev = device if device is not None else tensors[0].device
    return torch.tensor([t.data_ptr() for t in tensors], dtype=torch.int64, device=dev)
