"""Binding of libkmq: same names as the C entry points, argument marshalling
only.  Every step of the layer runs in the CUDA library; there is no Python or
CPU implementation behind these calls, and loading fails loudly when the shared
library has not been built.

The entry points that enqueue GPU work are functions of the extension module
``_kmq_native`` (csrc/kmq_python.cpp), because a decode call is so short that
marshalling in Python would cost more than the call; the host-side helpers go
through ctypes.

Tensor arguments are ``torch`` CUDA tensors (used for device memory only) or
raw integer device addresses; ``stream`` defaults to torch's current stream.
Every entry point returns the status and, unless ``check=False``, raises
``KmqError`` when it is not 0.
"""
from __future__ import annotations

import ctypes
import importlib.machinery
import importlib.util
import os
import sysconfig

_PKG_DIR = os.path.dirname(os.path.abspath(__file__))
_LIB_PATH = os.path.join(_PKG_DIR, "libkmq.so")
_NATIVE_PATH = os.path.join(_PKG_DIR, "_kmq_native" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
_lib = None
_native = None

KMQ_OK = 0
KMQ_ERR_NULL, KMQ_ERR_BITS, KMQ_ERR_SHAPE, KMQ_ERR_ALIGN = 1, 2, 3, 4
KMQ_ERR_WORKSPACE, KMQ_ERR_LAYOUT, KMQ_ERR_CUDA = 5, 6, 7
KMQ_ERR_SCRATCH_LIMIT = 8
KMQ_LAYOUT_CANONICAL = 0
KMQ_LAYOUT_TUNED = 1
KMQ_LAYOUT_TABLE = 2
KMQ_SCALE_DIRECT, KMQ_SCALE_DEFERRED = 0, 1
KMQ_LAMBDA_ABSMAX, KMQ_LAMBDA_ABSMEAN = 0, 1
KMQ_DEVICE_ERROR_WAIT_TIMEOUT = 1
KMQ_DEVICE_ERROR_SMEM_WINDOW = 2

_i64, _int, _ptr, _sz = ctypes.c_int64, ctypes.c_int, ctypes.c_void_p, ctypes.c_size_t

# name -> (restype, argtypes); mirrors include/kmq.h
SIGNATURES = {
    "kmq_version": (_int, []),
    "kmq_status_string": (ctypes.c_char_p, [_int]),
    "kmq_packed_bytes": (_sz, [_i64, _i64, _int, _int]),
    "kmq_packed_word_index": (_i64, [_i64, _i64, _i64, _i64, _int, _int]),
    "kmq_packed_field_shift": (_int, [_int, _int, _int]),
    "kmq_packed_bit_index": (_i64, [_i64, _i64, _int, _i64, _i64, _int, _int]),
    "kmq_preferred_layout": (_int, [_i64, _i64, _int, _i64]),
    "kmq_workspace_bytes": (_sz, [_i64, _i64, _int, _i64, _int]),
    "kmq_linear_num_launches": (_int, [_i64, _i64, _int, _i64, _int]),
    "kmq_linear_variant": (ctypes.c_char_p, [_i64, _i64, _int, _i64, _int]),
    "kmq_pack": (_int, [_ptr, _i64, _i64, _int, _int, _ptr, _ptr]),
    "kmq_unpack": (_int, [_ptr, _i64, _i64, _int, _int, _ptr, _ptr]),
    "kmq_linear": (_int, [_ptr, _ptr, _ptr, _ptr, _i64, _i64, _int, _i64, _int, _ptr, _sz, _ptr]),
    "kmq_linear_host": (_int, [_ptr, _ptr, _ptr, _ptr, _i64, _i64, _int, _i64, _int, _ptr, _ptr, _ptr, _sz, _ptr]),
    "kmq_linear_static_scratch": (_int, [_ptr, _ptr, _ptr, _ptr, _i64, _i64, _int, _i64, _int, _ptr]),
    "kmq_static_scratch_capacity": (_sz, []),
    "kmq_linear_tcgen05": (_int, [_ptr, _ptr, _ptr, _ptr, _i64, _i64, _int, _i64, _ptr]),
    "kmq_device_error_flags": (_int, [_ptr]),
    "kmq_dequant_to_bf16": (_int, [_ptr, _ptr, _ptr, _i64, _i64, _int, _int, _ptr]),
    "kmq_block_packed_bytes": (_sz, [_i64, _i64, _int]),
    "kmq_block_pack": (_int, [_ptr, _i64, _i64, _int, _ptr, _ptr]),
    "kmq_block_linear": (_int, [_ptr, _ptr, _ptr, _ptr, _ptr, _i64, _i64, _int, _i64, _int, _ptr]),
    "kmq_block_dequant_to_bf16": (_int, [_ptr, _ptr, _ptr, _ptr, _i64, _i64, _int, _ptr]),
    "kmq_block_table_bytes": (_sz, [_i64, _i64, _int]),
    "kmq_block_table_index_offset": (_i64, [_i64, _i64, _i64, _i64, _int]),
    "kmq_block_table_scale_offset": (_i64, [_i64, _i64, _i64, _i64, _int]),
    "kmq_block_table_pack": (_int, [_ptr, _ptr, _i64, _i64, _int, _ptr, _ptr]),
    "kmq_block_table_unpack": (_int, [_ptr, _i64, _i64, _int, _ptr, _ptr, _ptr]),
    "kmq_block_table_workspace_bytes": (_sz, [_i64, _i64, _int]),
    "kmq_block_table_linear": (_int, [_ptr, _ptr, _ptr, _ptr, _i64, _i64, _int, _i64, _ptr, _sz, _ptr]),
    "kmq_kmeans_rows": (_int, [_ptr, _i64, _i64, _int, _int, _ptr, _ptr, _ptr]),
    "kmq_assign_pack": (_int, [_ptr, _ptr, _i64, _i64, _int, _int, _ptr, _ptr]),
    "kmq_quantize_rows": (_int, [_ptr, _i64, _i64, _int, _int, _int, _ptr, _ptr, _ptr]),
    "kmq_block_scales": (_int, [_ptr, _i64, _i64, _int, _ptr, _ptr]),
    "kmq_block_sample_count": (_i64, [_i64, _i64, _i64]),
    "kmq_block_sample": (_int, [_ptr, _ptr, _i64, _i64, _i64, _ptr, _ptr]),
    "kmq_block_assign_pack": (_int, [_ptr, _ptr, _ptr, _i64, _i64, _int, _ptr, _ptr]),
    "kmq_block_quantize": (_int, [_ptr, _i64, _i64, _int, _int, _int, _i64, _ptr, _ptr, _ptr, _ptr, _ptr]),
    "kmq_probe_launch": (_int, [_ptr]),
    "kmq_probe_read_out_bytes": (_sz, []),
    "kmq_probe_read": (_int, [_ptr, _sz, _ptr, _ptr]),
}


class KmqError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {status_string(status)} (status {status})")


def lib() -> ctypes.CDLL:
    """Load libkmq.so (once).  Raises if it is missing: there is no fallback."""
    global _lib
    if _lib is None:
        if not os.path.exists(_LIB_PATH):
            raise ImportError(
                f"{_LIB_PATH} not found: build it with "
                "`python -m paper_2602_15563_b200.build` (needs nvcc); libkmq has no CPU fallback")
        handle = ctypes.CDLL(_LIB_PATH)
        for name, (res, args) in SIGNATURES.items():
            fn = getattr(handle, name)
            fn.restype, fn.argtypes = res, args
        _lib = handle
    return _lib


def _load_native():
    """The extension module (once).  Raises if it is missing: there is no other way to these calls."""
    global _native
    if _native is None:
        if not os.path.exists(_NATIVE_PATH) or not os.path.exists(_LIB_PATH):
            raise ImportError(
                f"{_NATIVE_PATH} or {_LIB_PATH} not found: build them with "
                "`python -m paper_2602_15563_b200.build` (needs nvcc); libkmq has no CPU fallback")
        loader = importlib.machinery.ExtensionFileLoader("_kmq_native", _NATIVE_PATH)
        module = importlib.util.module_from_spec(importlib.util.spec_from_loader("_kmq_native", loader))
        loader.exec_module(module)
        module.set_error(KmqError)
        _native = module
    return _native


# Entry points that enqueue work, with their Python arguments; looked up in the extension module on first use.
#   kmq_pack(idx, N, K, bits, packed, layout=CANONICAL, ...)
#   kmq_unpack(packed, N, K, bits, idx, layout=CANONICAL, ...)
#   kmq_linear(packed, codebooks, x, y, N, K, bits, M, workspace=None, workspace_bytes=None, layout=CANONICAL, ...)
#   kmq_linear_host(packed, codebooks, x_host, y_host, N, K, bits, M, x_dev, y_dev, workspace=None,
#                   workspace_bytes=None, layout=CANONICAL, ...)
#   kmq_linear_static_scratch(packed, codebooks, x, y, N, K, bits, M, layout=CANONICAL, ...)
#   kmq_linear_tcgen05(packed, codebooks, x, y, N, K, bits, M, ...)
#   kmq_dequant_to_bf16(packed, codebooks, W, N, K, bits, layout=CANONICAL, ...)
#   kmq_block_pack(idx, N, K, bits, wq, ...)
#   kmq_block_linear(wq, scales, codebook, x, y, N, K, bits, M, scale_order=DEFERRED, ...)
#   kmq_block_dequant_to_bf16(wq, scales, codebook, W, N, K, bits, ...)
#   kmq_block_table_pack(wq, scales, N, K, bits, table, ...)
#   kmq_block_table_unpack(table, N, K, bits, wq, scales, ...)
#   kmq_block_table_linear(table, codebook, x, y, N, K, bits, M, workspace=None, workspace_bytes=0, ...)
#   kmq_kmeans_rows(W, N, K, bits, iters, codebooks, centroids=None, ...)
#   kmq_assign_pack(W, codebooks, N, K, bits, layout, packed, ...)
#   kmq_quantize_rows(W, N, K, bits, iters, layout, codebooks, packed, ...)
#   kmq_block_scales(W, N, K, lam, scales, ...)
#   kmq_block_sample(W, scales, N, K, samples, out, ...)
#   kmq_block_assign_pack(W, scales, codebook, N, K, bits, wq, ...)
#   kmq_block_quantize(W, N, K, bits, lam, iters, samples, scales, codebook, wq, sample_workspace, ...)
#   kmq_probe_launch(...)
#   kmq_probe_read(buf, nbytes, out, ...)
# "..." = stream=None, check=True.
_HOST_SIDE = ("kmq_device_error_flags",)
_ENQUEUE = frozenset(n for n, (_, args) in SIGNATURES.items()
                     if _ptr in args and n not in _HOST_SIDE)


def __getattr__(name):
    if name in _ENQUEUE:
        fn = getattr(_load_native(), name)
        globals()[name] = fn
        return fn
    raise AttributeError(f"module {__name__!r} has no attribute {name!r}")


def _check(status: int, where: str) -> None:
    if status != KMQ_OK:
        raise KmqError(status, where)


def status_string(status: int) -> str:
    return lib().kmq_status_string(int(status)).decode()


def kmq_version() -> int:
    return lib().kmq_version()


def kmq_packed_bytes(N, K, bits, layout=KMQ_LAYOUT_CANONICAL) -> int:
    return lib().kmq_packed_bytes(N, K, bits, layout)


def kmq_packed_word_index(n, j, N, K, bits, layout=KMQ_LAYOUT_CANONICAL) -> int:
    return lib().kmq_packed_word_index(n, j, N, K, bits, layout)


def kmq_packed_field_shift(i, bits, layout=KMQ_LAYOUT_CANONICAL) -> int:
    return lib().kmq_packed_field_shift(i, bits, layout)


def kmq_packed_bit_index(n, k, plane, N, K, bits, layout=KMQ_LAYOUT_CANONICAL) -> int:
    return lib().kmq_packed_bit_index(n, k, plane, N, K, bits, layout)


def kmq_preferred_layout(N, K, bits, M) -> int:
    return lib().kmq_preferred_layout(N, K, bits, M)


def kmq_workspace_bytes(N, K, bits, M, layout=KMQ_LAYOUT_CANONICAL) -> int:
    return lib().kmq_workspace_bytes(N, K, bits, M, layout)


def kmq_linear_num_launches(N, K, bits, M, layout=KMQ_LAYOUT_CANONICAL) -> int:
    return lib().kmq_linear_num_launches(N, K, bits, M, layout)


def kmq_linear_variant(N, K, bits, M, layout=KMQ_LAYOUT_CANONICAL) -> str:
    return lib().kmq_linear_variant(N, K, bits, M, layout).decode()


def kmq_static_scratch_capacity() -> int:
    return lib().kmq_static_scratch_capacity()


def kmq_device_error_flags() -> int:
    """Synchronise the device; return and clear the error word of the kernels (0 = no bounded wait ran out)."""
    flags = ctypes.c_uint(0)
    _check(lib().kmq_device_error_flags(ctypes.addressof(flags)), "kmq_device_error_flags")
    return flags.value


def kmq_probe_read_out_bytes() -> int:
    return lib().kmq_probe_read_out_bytes()


def kmq_block_packed_bytes(N, K, bits) -> int:
    return lib().kmq_block_packed_bytes(N, K, bits)


def kmq_block_sample_count(N, K, samples) -> int:
    return lib().kmq_block_sample_count(N, K, samples)


def kmq_block_table_bytes(N, K, bits) -> int:
    return lib().kmq_block_table_bytes(N, K, bits)


def kmq_block_table_index_offset(n, k, N, K, bits) -> int:
    return lib().kmq_block_table_index_offset(n, k, N, K, bits)


def kmq_block_table_scale_offset(n, k, N, K, bits) -> int:
    return lib().kmq_block_table_scale_offset(n, k, N, K, bits)


def kmq_block_table_workspace_bytes(N, K, bits) -> int:
    return lib().kmq_block_table_workspace_bytes(N, K, bits)


