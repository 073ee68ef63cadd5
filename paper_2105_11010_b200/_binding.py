"""Binding with the same names as the C ABI in ``include/sparq.h``.

Argument marshalling only.  Tensors must already live on the CUDA device (the
raw ``data_ptr`` is handed to the library) and work is enqueued on torch's
current stream unless a stream is given.  The calls of a forward pass go through the
native module ``_native`` (``csrc/sparq_py.cpp``), which takes their arguments by position;
diagnostics and set-up calls use ctypes.
"""
from __future__ import annotations

import ctypes
import os
from dataclasses import dataclass
from typing import Optional

import torch

MODE_NONE, MODE_BSPARQ, MODE_VSPARQ = 0, 1, 2
ROUND_TRUNCATE, ROUND_NEAREST = 0, 1
SET_5OPT, SET_3OPT, SET_2OPT, SET_6OPT, SET_7OPT = 0x1F, 0x15, 0x11, 0x3F, 0x7F

_PKG = os.path.dirname(os.path.abspath(__file__))
_LIB_PATH = os.path.join(_PKG, "libsparq_b200.so")


class SparqError(RuntimeError):
    def __init__(self, code: int, text: str):
        super().__init__(f"sparq error {code}: {text}")
        self.code = code


class _CParams(ctypes.Structure):
    _fields_ = [("mode", ctypes.c_int32), ("window_bits", ctypes.c_int32),
                ("placement_mask", ctypes.c_uint32), ("rounding", ctypes.c_int32)]


class _CEpilogue(ctypes.Structure):
    _fields_ = [("scale", ctypes.c_void_p), ("bias", ctypes.c_void_p),
                ("relu", ctypes.c_int32), ("inv_out_scale", ctypes.c_float),
                ("acc_out", ctypes.c_void_p), ("f32_out", ctypes.c_void_p),
                ("u8_out", ctypes.c_void_p), ("next_transform", ctypes.POINTER(_CParams)),
                ("residual", ctypes.c_void_p), ("residual_scale", ctypes.c_float)]


@dataclass(frozen=True)
class SparqParams:
    """Mirror of ``sparq_params``."""
    mode: int = MODE_VSPARQ
    window_bits: int = 4
    placement_mask: int = SET_5OPT
    rounding: int = ROUND_NEAREST

    def _c(self) -> _CParams:
        return _CParams(self.mode, self.window_bits, self.placement_mask, self.rounding)


_lib: Optional[ctypes.CDLL] = None


def library_path() -> str:
    return _LIB_PATH


def load_library() -> ctypes.CDLL:
    """Loads the built C-ABI library; raises if it has not been built."""
    global _lib
    if _lib is None:
        if not os.path.exists(_LIB_PATH):
            raise ImportError(
                f"{_LIB_PATH} is missing: build it with `python -m paper_2105_11010_b200.build` "
                "(needs nvcc); this package has no CPU fallback")
        L = ctypes.CDLL(_LIB_PATH)
        vp, i32, i64, sz = ctypes.c_void_p, ctypes.c_int, ctypes.c_int64, ctypes.c_size_t
        L.sparq_quantize.argtypes = [vp, vp, sz, sz, ctypes.POINTER(_CParams), vp]
        L.sparq_quantize.restype = i32
        L.sparq_gemm_s8.argtypes = [vp, i64, vp, i64, i64, i64, i64,
                                    ctypes.POINTER(_CParams), ctypes.POINTER(_CEpilogue), vp]
        L.sparq_gemm_s8.restype = i32
        L.sparq_conv2d_nhwc_s8.argtypes = [vp, i32, i32, i32, i32, vp, i32, i32, i32,
                                           i32, i32, i32, i32,
                                           ctypes.POINTER(_CParams), ctypes.POINTER(_CEpilogue), vp]
        L.sparq_conv2d_nhwc_s8.restype = i32
        L.sparq_packed_ctrl_bits.argtypes = [ctypes.POINTER(_CParams)]
        L.sparq_packed_ctrl_bits.restype = i32
        L.sparq_pack.argtypes = [vp, sz, sz, ctypes.POINTER(_CParams), vp, vp, vp]
        L.sparq_pack.restype = i32
        L.sparq_unpack.argtypes = [vp, vp, sz, sz, ctypes.POINTER(_CParams), vp, vp]
        L.sparq_unpack.restype = i32
        L.sparq_absmax.argtypes = [vp, i32, sz, vp, vp]
        L.sparq_absmax.restype = i32
        L.sparq_quantize_act_u8.argtypes = [vp, i32, sz, vp, vp, vp]
        L.sparq_quantize_act_u8.restype = i32
        L.sparq_quantize_weight_s8.argtypes = [vp, i64, i64, vp, vp, vp]
        L.sparq_quantize_weight_s8.restype = i32
        L.sparq_sparse24_expanded_k.argtypes = [i64, ctypes.POINTER(_CParams)]
        L.sparq_sparse24_expanded_k.restype = i64
        L.sparq_sparse24_expand_weights.argtypes = [vp, vp, i64, i64, ctypes.POINTER(_CParams), vp, vp]
        L.sparq_sparse24_expand_weights.restype = i32
        L.sparq_sparse24_expand_activations.argtypes = [vp, sz, sz, ctypes.POINTER(_CParams), vp, vp]
        L.sparq_sparse24_expand_activations.restype = i32
        L.sparq_gemm_s8_sparse24.argtypes = [vp, vp, i64, i64, i64, ctypes.POINTER(_CParams),
                                             ctypes.POINTER(_CEpilogue), vp, vp]
        L.sparq_gemm_s8_sparse24.restype = i32
        L.sparq_quantize_host.argtypes = L.sparq_quantize.argtypes
        L.sparq_quantize_host.restype = i32
        L.sparq_gemm_s8_host.argtypes = L.sparq_gemm_s8.argtypes
        L.sparq_gemm_s8_host.restype = i32
        L.sparq_conv2d_nhwc_s8_host.argtypes = L.sparq_conv2d_nhwc_s8.argtypes
        L.sparq_conv2d_nhwc_s8_host.restype = i32
        L.sparq_gemm_s8_static.argtypes = L.sparq_gemm_s8.argtypes
        L.sparq_gemm_s8_static.restype = i32
        L.sparq_selftest_wait_timeout.argtypes = [i64, i32, vp, vp]
        L.sparq_selftest_wait_timeout.restype = i32
        L.sparq_selftest_mma_rate.argtypes = [i32, i32, vp, vp]
        L.sparq_selftest_mma_rate.restype = i32
        L.sparq_selftest_form.argtypes = [i32] * 11 + [ctypes.POINTER(_CParams), i32]
        L.sparq_selftest_form.restype = i32
        L.sparq_check.argtypes = [vp]
        L.sparq_check.restype = i32
        L.sparq_last_error.argtypes = []
        L.sparq_last_error.restype = ctypes.c_char_p
        L.sparq_shutdown.argtypes = []
        L.sparq_shutdown.restype = i32
        _lib = L
    return _lib


def load_native():
    """The native call module; raises if it has not been built."""
    load_library()
    try:
        from . import _native
    except ImportError as e:
        raise ImportError("the native call module of this package is missing or does not load: build it with "
                          "`python -m paper_2105_11010_b200.build`") from e
    return _native


class _LazyNative:
    """Stands for the native module until the first call, so that the package imports unbuilt."""

    def __getattr__(self, name):
        global _native
        _native = load_native()
        return getattr(_native, name)


_native = _LazyNative()


def _stream_ptr(stream) -> Optional[int]:
    if stream is None:
        stream = torch.cuda.current_stream()
    if isinstance(stream, int):
        return stream or None
    return stream.cuda_stream or None


def _dev(t: Optional[torch.Tensor], dtype, name: str) -> Optional[int]:
    if t is None:
        return None
    if not t.is_cuda:
        raise ValueError(f"{name} must be a CUDA tensor")
    if t.dtype != dtype:
        raise ValueError(f"{name} must have dtype {dtype}, got {t.dtype}")
    if not t.is_contiguous():
        raise ValueError(f"{name} must be contiguous")
    return t.data_ptr() or None


def _raise(code: int) -> None:
    if code != 0:
        raise SparqError(code, sparq_last_error())


def sparq_last_error() -> str:
    return load_library().sparq_last_error().decode()


def sparq_check(stream=None) -> None:
    _raise(load_library().sparq_check(_stream_ptr(stream)))


def sparq_selftest_wait_timeout(limit_cycles: int, report: torch.Tensor, use_static_word: bool = False,
                                stream=None) -> None:
    """Diagnostic launch whose bounded wait runs out; ``report`` is 4 int32/uint32 words on the device."""
    if report.numel() < 4 or report.element_size() != 4 or not report.is_cuda:
        raise ValueError("report must hold four 32-bit words on the device")
    _raise(load_library().sparq_selftest_wait_timeout(int(limit_cycles), int(bool(use_static_word)),
                                                      report.data_ptr(), _stream_ptr(stream)))


def sparq_selftest_mma_rate(bn: int, iters: int, cycles_out: torch.Tensor, stream=None) -> int:
    """MMA-only loop on every SM; ``cycles_out`` (int64, one per SM, device) receives each CTA's cycles.
    Returns the number of CTAs launched."""
    if cycles_out.dtype != torch.int64 or not cycles_out.is_cuda or cycles_out.numel() < 256:
        raise ValueError("cycles_out must be an int64 device tensor of at least 256 elements")
    rc = load_library().sparq_selftest_mma_rate(int(bn), int(iters), cycles_out.data_ptr(), _stream_ptr(stream))
    if rc < 0:
        _raise(rc)
    return rc


FORM_FULL, FORM_SMALL, FORM_WINDOW_RESIDENT, FORM_WINDOW_STREAMED, FORM_TRANSFORM_FIRST = range(5)


def sparq_selftest_form(x_shape, w_shape, stride, pad, params: SparqParams, sms: int = 148) -> int:
    """The form (``FORM_*``) that a convolution of this shape takes; host arithmetic only."""
    n, h, w, c = x_shape
    cout, r, s, _ = w_shape
    p = params._c()
    rc = load_library().sparq_selftest_form(n, h, w, c, cout, r, s, stride[0], stride[1], pad[0], pad[1], ctypes.byref(p), sms)
    if rc < 0:
        _raise(rc)
    return rc


def sparq_shutdown() -> None:
    _raise(load_library().sparq_shutdown())


def sparq_quantize(inp: torch.Tensor, out: torch.Tensor, rows: int, row_len: int,
                   params: SparqParams, stream=None) -> None:
    """``out = T(inp)`` for ``rows`` rows of ``row_len`` uint8 activations."""
    rc = _native.quantize(inp, out, rows, row_len, params, stream)
    if rc:
        _raise(rc)


def sparq_gemm_s8(A: torch.Tensor, B: torch.Tensor, params: SparqParams, *,
                  scale: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None,
                  relu: bool = False, inv_out_scale: float = 1.0,
                  acc_out: Optional[torch.Tensor] = None, f32_out: Optional[torch.Tensor] = None,
                  u8_out: Optional[torch.Tensor] = None,
                  next_transform: Optional[SparqParams] = None,
                  residual: Optional[torch.Tensor] = None, residual_scale: float = 0.0, stream=None) -> None:
    """``acc = T(A) @ B^T`` with A (M, K) uint8 and B (N, K) int8, then the epilogue."""
    rc = _native.gemm(A, B, params, scale, bias, relu, inv_out_scale, acc_out, f32_out, u8_out,
                      next_transform, residual, residual_scale, stream)
    if rc:
        _raise(rc)


def sparq_conv2d_nhwc_s8(x: torch.Tensor, w: torch.Tensor, stride, pad, params: SparqParams, *,
                         scale: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None,
                         relu: bool = False, inv_out_scale: float = 1.0,
                         acc_out: Optional[torch.Tensor] = None, f32_out: Optional[torch.Tensor] = None,
                         u8_out: Optional[torch.Tensor] = None,
                  next_transform: Optional[SparqParams] = None,
                  residual: Optional[torch.Tensor] = None, residual_scale: float = 0.0, stream=None) -> None:
    """Fused convolution of NHWC uint8 ``x`` with [cout][r][s][c] int8 ``w``."""
    rc = _native.conv2d(x, w, stride, pad, params, scale, bias, relu, inv_out_scale, acc_out, f32_out, u8_out,
                        next_transform, residual, residual_scale, stream)
    if rc:
        _raise(rc)


# ---- packed stream ------------------------------------------------------------------------

def sparq_packed_ctrl_bits(params: SparqParams) -> int:
    """Control bits per pair of the packed stream for these parameters."""
    p = params._c()
    rc = load_library().sparq_packed_ctrl_bits(ctypes.byref(p))
    if rc < 0:
        _raise(rc)
    return rc


def sparq_pack(inp: torch.Tensor, params: SparqParams, data: torch.Tensor, ctrl: torch.Tensor, stream=None) -> None:
    """Packed stream of ``inp`` (rows along the last axis) into the caller's ``data``
    (numel / 16 * 2 * window_bits bytes) and ``ctrl`` (numel / 16 * ctrl_bits bytes) planes."""
    rc = _native.pack(inp, params, data, ctrl, stream)
    if rc:
        _raise(rc)


def sparq_unpack(data: torch.Tensor, ctrl: torch.Tensor, params: SparqParams, out: torch.Tensor, stream=None) -> None:
    """``out`` (rows along the last axis) = T(x) of the packed stream."""
    rc = _native.unpack(out, params, data, ctrl, stream)
    if rc:
        _raise(rc)


# ---- uniform min-max quantization front end -----------------------------------------------

DTYPE_F32, DTYPE_BF16 = 0, 1


def sparq_absmax(x: torch.Tensor, max_inout: torch.Tensor, stream=None) -> None:
    """``max_inout[0] = max(max_inout[0], max |x|)`` on the device (float32, 1 element)."""
    rc = _native.absmax(x, max_inout, stream)
    if rc:
        _raise(rc)


def sparq_quantize_act_u8(x: torch.Tensor, max_dev: torch.Tensor, out: torch.Tensor, stream=None) -> None:
    """Unsigned symmetric per-layer quantization of ``x`` onto [0, max] in 255 steps."""
    rc = _native.quantize_act(x, max_dev, out, stream)
    if rc:
        _raise(rc)


def sparq_quantize_weight_s8(w: torch.Tensor, out: torch.Tensor, scale_out: torch.Tensor, stream=None) -> None:
    """Signed symmetric per-kernel quantization of float32 ``w`` (kernels along axis 0)."""
    rc = _native.quantize_weight(w, out, scale_out, stream)
    if rc:
        _raise(rc)


# ---- 2:4 sparse weights ---------------------------------------------------------------------

def sparq_sparse24_expanded_k(K: int, params: SparqParams) -> int:
    p = params._c()
    rc = load_library().sparq_sparse24_expanded_k(K, ctypes.byref(p))
    if rc < 0:
        _raise(int(rc))
    return int(rc)


def sparq_sparse24_expand_weights(vals: torch.Tensor, pos: torch.Tensor, params: SparqParams, w_exp: torch.Tensor,
                                  stream=None) -> None:
    """Compressed 2:4 weights (vals, pos: (N, K/2)) -> ``w_exp`` (N, K')."""
    N = vals.shape[0]
    K = 2 * (vals.numel() // N) if N else 0
    if pos.numel() != vals.numel() or w_exp.numel() < N * sparq_sparse24_expanded_k(K, params):
        raise ValueError("pos / w_exp size does not match vals")
    p = params._c()
    _raise(load_library().sparq_sparse24_expand_weights(_dev(vals, torch.int8, "vals"), _dev(pos, torch.uint8, "pos"),
                                                        N, K, ctypes.byref(p), _dev(w_exp, torch.int8, "w_exp"),
                                                        _stream_ptr(stream)))


def sparq_sparse24_expand_activations(A: torch.Tensor, params: SparqParams, a_exp: torch.Tensor, stream=None) -> None:
    """Activations (rows along the last axis, K) -> ``a_exp`` with K' per row."""
    rc = _native.expand_activations(A, params, a_exp, stream)
    if rc:
        _raise(rc)


def sparq_gemm_s8_sparse24(A: torch.Tensor, w_exp: torch.Tensor, params: SparqParams, *,
                           workspace: Optional[torch.Tensor] = None,
                           scale: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None,
                           relu: bool = False, inv_out_scale: float = 1.0,
                           acc_out: Optional[torch.Tensor] = None, f32_out: Optional[torch.Tensor] = None,
                           u8_out: Optional[torch.Tensor] = None, stream=None) -> None:
    """``acc[m][j] = sum_g T2(selected pair) . (v0, v1)`` for 2:4 weights expanded by
    :func:`sparq_sparse24_expand_weights`, then the epilogue."""
    rc = _native.gemm_sparse24(A, w_exp, params, workspace, scale, bias, relu, inv_out_scale, acc_out, f32_out, u8_out,
                               None, None, 0.0, stream)
    if rc:
        _raise(rc)


# ---- host-buffer forms ------------------------------------------------------------------

def sparq_quantize_host(inp: torch.Tensor, out: torch.Tensor, rows: int, row_len: int,
                        params: SparqParams, stream=None) -> None:
    """Host-buffer form of :func:`sparq_quantize`; returns after the result is in ``out``."""
    rc = _native.quantize_host(inp, out, rows, row_len, params, stream)
    if rc:
        _raise(rc)


def sparq_gemm_s8_host(A: torch.Tensor, B: torch.Tensor, params: SparqParams, *,
                       scale: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None,
                       relu: bool = False, inv_out_scale: float = 1.0,
                       acc_out: Optional[torch.Tensor] = None, f32_out: Optional[torch.Tensor] = None,
                       u8_out: Optional[torch.Tensor] = None,
                  residual: Optional[torch.Tensor] = None, residual_scale: float = 0.0, stream=None) -> None:
    """Host-buffer form of :func:`sparq_gemm_s8`: ``A`` and the outputs are CPU tensors."""
    rc = _native.gemm_host(A, B, params, scale, bias, relu, inv_out_scale, acc_out, f32_out, u8_out,
                           None, residual, residual_scale, stream)
    if rc:
        _raise(rc)


def sparq_conv2d_nhwc_s8_host(x: torch.Tensor, w: torch.Tensor, stride, pad, params: SparqParams, *,
                              scale: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None,
                              relu: bool = False, inv_out_scale: float = 1.0,
                              acc_out: Optional[torch.Tensor] = None, f32_out: Optional[torch.Tensor] = None,
                              u8_out: Optional[torch.Tensor] = None,
                  residual: Optional[torch.Tensor] = None, residual_scale: float = 0.0, stream=None) -> None:
    """Host-buffer form of :func:`sparq_conv2d_nhwc_s8`: ``x`` and the outputs are CPU tensors."""
    rc = _native.conv2d_host(x, w, stride, pad, params, scale, bias, relu, inv_out_scale, acc_out, f32_out, u8_out,
                             None, residual, residual_scale, stream)
    if rc:
        _raise(rc)


STATIC_SCRATCH_BYTES = 8 << 20


def sparq_gemm_s8_static(A: torch.Tensor, B: torch.Tensor, params: SparqParams, *,
                         scale: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None,
                         relu: bool = False, inv_out_scale: float = 1.0,
                         acc_out: Optional[torch.Tensor] = None, f32_out: Optional[torch.Tensor] = None,
                         u8_out: Optional[torch.Tensor] = None,
                  next_transform: Optional[SparqParams] = None,
                  residual: Optional[torch.Tensor] = None, residual_scale: float = 0.0, stream=None) -> None:
    """``sparq_gemm_s8`` for hosts that must not allocate device memory once running
    (all free memory already belongs to a framework's pool, or an allocation's
    device-wide synchronization is not acceptable).  Same result, computed as transform
    kernel + plain GEMM with the transformed activations in a fixed scratch array inside
    the library (``M * K <= STATIC_SCRATCH_BYTES``).  Synchronous; one call at a time per
    device.  The first call on a device performs the address look-up: make it before any
    stream capture."""
    rc = _native.gemm_static(A, B, params, scale, bias, relu, inv_out_scale, acc_out, f32_out, u8_out,
                             next_transform, residual, residual_scale, stream)
    if rc:
        _raise(rc)
