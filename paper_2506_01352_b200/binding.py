"""Binding of the C ABI in include/tahq.h (argument marshalling only): the codec calls themselves through the
extension module ``_call``, everything else through ctypes.

Every step of encode and decode runs in the CUDA kernels of ``libtahq.so``; PyTorch is used here
for device memory and streams.  There is no CPU fallback: importing this module without the built
library raises.
"""
from __future__ import annotations

import ctypes as C
import os
from dataclasses import dataclass

import torch

from . import build as _build

F32, BF16 = 0, 1
OK = 0
DEV_OK, DEV_BAD_HEADER, DEV_BAD_BITMAP, DEV_TIMEOUT, DEV_INTERNAL = 0, 1, 2, 4, 8


class _Params(C.Structure):
    _fields_ = [
        ("struct_size", C.c_uint32), ("dtype", C.c_uint32), ("tokens", C.c_uint64), ("hidden", C.c_uint32),
        ("group_tokens", C.c_uint32), ("tile", C.c_uint32), ("budget_millibits", C.c_uint32),
        ("tau", C.c_float), ("eps_l1", C.c_float), ("eps_log", C.c_float), ("eps_ratio", C.c_float),
        ("rounding", C.c_uint32), ("seed", C.c_uint64), ("alloc_tile", C.c_uint32),
    ]


class _Layout(C.Structure):
    _fields_ = [
        ("n_tiles", C.c_uint64), ("n_groups", C.c_uint64), ("tiles_per_group", C.c_uint64), ("k_hi", C.c_uint64),
        ("lo_bits", C.c_uint32), ("hi_bits", C.c_uint32), ("off_bitmap", C.c_uint64),
        ("off_scale_zero", C.c_uint64), ("off_pivot", C.c_uint64), ("off_payload", C.c_uint64),
        ("payload_bytes", C.c_uint64), ("total_bytes", C.c_uint64),
    ]


class _Kept:
    """Parameters whose C structure is laid out once, not on every call.

    The bytes lie in a box; a change of a field puts an empty box in its place.  A thread that lays the structure out while
    another one changes a field fills the box that it took before it read the fields, so what it read can be kept only as
    long as it is current.  The box is no part of the object's state: not of ``vars()``, of copies or of pickles.  (A value
    that is put into ``vars()`` behind the object's back is seen after the next change of a field.)
    """

    __slots__ = ("_box",)

    def __setattr__(self, name, value):
        object.__setattr__(self, name, value)
        _set_box(self, [None])

    def __delattr__(self, name):   # (the field has its default again)
        object.__delattr__(self, name)
        _set_box(self, [None])

    def __getstate__(self):
        return self.__dict__

    def __setstate__(self, state):
        self.__dict__.update(state)
        _set_box(self, [None])

    def raw(self) -> bytes:
        """The bytes of the C structure."""
        box = self._box
        b = box[0]
        if b is None:
            b = box[0] = bytes(self.c())
        return b


_set_box = _Kept._box.__set__


@dataclass
class Params(_Kept):
    """tahq_params: one boundary tensor [tokens x hidden]; G = tile, S = group_tokens (paper notation)."""

    tokens: int
    hidden: int
    dtype: int = F32
    group_tokens: int = 0
    tile: int = 64
    budget_millibits: int = 3800
    tau: float = 2.0
    eps_l1: float = 1e-8
    eps_log: float = 1e-8
    eps_ratio: float = 1e-8
    rounding: int = 0
    seed: int = 0
    alloc_tile: int = 0

    def c(self) -> _Params:
        return _Params(C.sizeof(_Params), self.dtype, self.tokens, self.hidden, self.group_tokens, self.tile,
                       self.budget_millibits, self.tau, self.eps_l1, self.eps_log, self.eps_ratio,
                       self.rounding, self.seed, self.alloc_tile)


class TahqError(RuntimeError):
    def __init__(self, code: int):
        self.code = code
        super().__init__(f"tahq: {status_string(code)} ({code})")


class _QParams(C.Structure):
    _fields_ = [("struct_size", C.c_uint32), ("dtype", C.c_uint32), ("tokens", C.c_uint64), ("hidden", C.c_uint32),
                ("bits", C.c_uint32), ("per_tensor", C.c_uint32), ("prescale", C.c_float)]


@dataclass
class QNaiveParams(_Kept):
    """Fixed-point gradient compressor (Algorithm 1 line 6): b bits, per-token or per-tensor scale, pre-scale c."""

    tokens: int
    hidden: int
    dtype: int = F32
    bits: int = 8
    per_tensor: int = 0
    prescale: float = 1.0

    def c(self) -> _QParams:
        return _QParams(C.sizeof(_QParams), self.dtype, self.tokens, self.hidden, self.bits, self.per_tensor,
                        self.prescale)


EXPORTS = ["tahq_packed_bound", "tahq_packed_layout", "tahq_workspace_bound", "tahq_encode", "tahq_decode",
           "tahq_encode_noalloc",
           "tahq_qnaive_packed_bound", "tahq_qnaive_workspace_bound", "tahq_qnaive_encode", "tahq_qnaive_decode",
           "tahq_selftest_wait_timeout",
           "tahq_status_string", "tahq_last_launch_count", "tahq_profile", "tahq_profile_read", "tahq_trace"]

_lib = None


def lib() -> C.CDLL:
    """Load libtahq.so (built in-tree).  Raises if it is missing: there is no other implementation."""
    global _lib
    if _lib is None:
        if not os.path.exists(_build.LIB):
            raise ImportError(f"{_build.LIB} is not built; run `python -c 'import __graft_entry__ as g; g.build()'`")
        L = C.CDLL(_build.LIB)
        pp = C.POINTER(_Params)
        L.tahq_packed_bound.argtypes = [pp]
        L.tahq_packed_bound.restype = C.c_size_t
        L.tahq_packed_layout.argtypes = [pp, C.POINTER(_Layout)]
        L.tahq_packed_layout.restype = C.c_int
        L.tahq_workspace_bound.argtypes = [pp]
        L.tahq_workspace_bound.restype = C.c_size_t
        L.tahq_encode.argtypes = [pp, C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p, C.c_size_t, C.c_void_p]
        L.tahq_encode.restype = C.c_int
        L.tahq_encode_noalloc.argtypes = [pp, C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p]
        L.tahq_encode_noalloc.restype = C.c_int
        L.tahq_decode.argtypes = [pp, C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p]
        L.tahq_decode.restype = C.c_int
        L.tahq_status_string.argtypes = [C.c_int]
        L.tahq_status_string.restype = C.c_char_p
        L.tahq_last_launch_count.argtypes = []
        L.tahq_last_launch_count.restype = C.c_int
        L.tahq_trace.argtypes = [C.c_void_p]
        L.tahq_trace.restype = None
        L.tahq_profile.argtypes = [C.c_int]
        L.tahq_profile.restype = None
        L.tahq_profile_read.argtypes = [C.c_char_p, C.POINTER(C.c_float), C.c_int]
        L.tahq_profile_read.restype = C.c_int
        qp = C.POINTER(_QParams)
        L.tahq_qnaive_packed_bound.argtypes = [qp]
        L.tahq_qnaive_packed_bound.restype = C.c_size_t
        L.tahq_qnaive_workspace_bound.argtypes = [qp]
        L.tahq_qnaive_workspace_bound.restype = C.c_size_t
        L.tahq_qnaive_encode.argtypes = [qp, C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p, C.c_size_t, C.c_void_p]
        L.tahq_qnaive_encode.restype = C.c_int
        L.tahq_qnaive_decode.argtypes = [qp, C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p]
        L.tahq_qnaive_decode.restype = C.c_int
        L.tahq_selftest_wait_timeout.argtypes = [C.c_void_p, C.c_size_t, C.c_void_p]
        L.tahq_selftest_wait_timeout.restype = C.c_int
        _lib = L
    return _lib


_call = None


def call():
    """The extension module with the codec calls.  Raises if it or the library is missing."""
    global _call
    if _call is None:
        lib()
        if not os.path.exists(_build.CALL):
            raise ImportError(f"{_build.CALL} is not built; run `python -c 'import __graft_entry__ as g; g.build()'`")
        from . import _call as m
        _call = m
    return _call


def status_string(code: int) -> str:
    return lib().tahq_status_string(int(code)).decode()


def packed_bound(p: Params) -> int:
    pc = p.c()
    return int(lib().tahq_packed_bound(C.byref(pc)))


def workspace_bound(p: Params) -> int:
    pc = p.c()
    return int(lib().tahq_workspace_bound(C.byref(pc)))


def packed_layout(p: Params) -> dict:
    pc, out = p.c(), _Layout()
    rc = lib().tahq_packed_layout(C.byref(pc), C.byref(out))
    if rc != OK:
        raise TahqError(rc)
    return {k: int(getattr(out, k)) for k, _ in _Layout._fields_}


def last_launch_count() -> int:
    return int(lib().tahq_last_launch_count())


def profile(enable: bool) -> None:
    """Switch the library's per-kernel event timing on or off."""
    lib().tahq_profile(1 if enable else 0)


def profile_read(max_records: int = 65536):
    """[(kernel name, milliseconds), ...] of the launches recorded since profile(True); synchronises."""
    names = C.create_string_buffer(32 * max_records)
    ms = (C.c_float * max_records)()
    n = lib().tahq_profile_read(names, ms, max_records)
    return [(names.raw[32 * i:32 * i + 32].split(b"\0")[0].decode(), float(ms[i])) for i in range(n)]


def trace(buf: "torch.Tensor | None") -> None:
    """Switch the kernel timeline on (buf: 64 int64 words on the device, preset by `trace_reset`) or off (None)."""
    lib().tahq_trace(None if buf is None else buf.data_ptr())


def trace_reset(buf: torch.Tensor) -> None:
    """Preset a timeline buffer: words 4k and 4k+1 to all-ones (minima), 4k+2 to zero (maximum)."""
    v = torch.full((16, 4), -1, dtype=torch.int64)
    v[:, 2] = 0
    buf.copy_(v.reshape(-1).to(buf.device))


# The current stream as a number.  torch.cuda.current_stream() builds an object around it, in three microseconds; the two
# functions that do without are private, so a torch that lacks one takes the public way.  The tensors of a call exist, so CUDA
# is initialised.
_device = getattr(torch._C, "_cuda_getDevice", torch.cuda.current_device)
_raw_stream = getattr(torch._C, "_cuda_getCurrentRawStream", lambda device: torch.cuda.current_stream(device).cuda_stream)


def tahq_encode(p: Params, d_in: int, d_packed: int, packed_cap: int, d_ws: int, ws_cap: int, stream: int) -> int:
    """Raw call: device addresses as integers, returns the tahq_status."""
    return (_call or call()).encode(p.raw(), d_in, d_packed, packed_cap, d_ws, ws_cap, stream)


NOALLOC_SCRATCH_BYTES = 8 << 20
ERR_TOO_LARGE = 6


def tahq_encode_noalloc(p: Params, d_in: int, d_packed: int, packed_cap: int, stream: int) -> int:
    """Raw call of the workspace-free encode: scratch comes from the library's built-in 8 MiB buffer.

    For callers that hold device pointers but cannot allocate (no allocator of their own, memory
    carved up in advance, or a place where an allocation would synchronise the device).  Returns the
    tahq_status; ERR_TOO_LARGE when workspace_bound(p) exceeds NOALLOC_SCRATCH_BYTES.  Calls on one
    device share the buffer, so calls that could overlap on the GPU must be ordered by the caller.
    """
    pc = p.c()
    return int(lib().tahq_encode_noalloc(C.byref(pc), d_in, d_packed, packed_cap, stream))


def tahq_decode(p: Params, d_packed: int, packed_bytes: int, d_out: int, d_ws: int, ws_cap: int, stream: int) -> int:
    return (_call or call()).decode(p.raw(), d_packed, packed_bytes, d_out, d_ws, ws_cap, stream)


def params_for(x: torch.Tensor, **kw) -> Params:
    if x.dim() != 2:
        raise ValueError("expected a [tokens x hidden] tensor")
    dt = {torch.float32: F32, torch.bfloat16: BF16}[x.dtype]
    return Params(tokens=x.shape[0], hidden=x.shape[1], dtype=dt, **kw)


def alloc_packed(p: Params, device="cuda") -> torch.Tensor:
    return torch.empty(packed_bound(p), dtype=torch.uint8, device=device)


def alloc_workspace(p: Params, device="cuda") -> torch.Tensor:
    return torch.empty(workspace_bound(p), dtype=torch.uint8, device=device)


def encode(p: Params, x: torch.Tensor, packed: torch.Tensor | None = None, ws: torch.Tensor | None = None,
           stream=None) -> torch.Tensor:
    """Encode a contiguous CUDA tensor; returns the packed uint8 buffer (asynchronous on the stream)."""
    if not (x.is_cuda and x.is_contiguous()):
        raise ValueError("x must be a contiguous CUDA tensor")
    made = packed is None or ws is None
    packed = alloc_packed(p, x.device) if packed is None else packed
    ws = alloc_workspace(p, x.device) if ws is None else ws
    if stream is not None and made:   # buffers made here belong to torch's current stream: tell the allocator who uses them
        packed.record_stream(stream)
        ws.record_stream(stream)
    rc = (_call or call()).encode(p._box[0] or p.raw(), x.data_ptr(), packed.data_ptr(), packed.numel(), ws.data_ptr(),
                                  ws.numel(), _raw_stream(_device()) if stream is None else stream.cuda_stream)
    if rc != OK:
        raise TahqError(rc)
    return packed


def decode(p: Params, packed: torch.Tensor, out: torch.Tensor | None = None, ws: torch.Tensor | None = None,
           stream=None) -> torch.Tensor:
    if out is None:
        out = torch.empty(p.tokens, p.hidden, dtype=torch.float32 if p.dtype == F32 else torch.bfloat16,
                          device=packed.device)
    made_ws = ws is None
    ws = alloc_workspace(p, packed.device) if ws is None else ws
    if stream is not None:
        if made_ws:
            ws.record_stream(stream)
        out.record_stream(stream)
    rc = (_call or call()).decode(p._box[0] or p.raw(), packed.data_ptr(), packed.numel(), out.data_ptr(), ws.data_ptr(),
                                  ws.numel(), _raw_stream(_device()) if stream is None else stream.cuda_stream)
    if rc != OK:
        raise TahqError(rc)
    return out


def device_status(ws: torch.Tensor) -> int:
    """Device status word of the last call that used this workspace (synchronises)."""
    return int(ws[:4].view(torch.int32).item())


# ---------------------------------------------------------------- fixed-point gradient compressor
def qnaive_packed_bound(p: QNaiveParams) -> int:
    return int(lib().tahq_qnaive_packed_bound(C.byref(p.c())))


def qnaive_workspace_bound(p: QNaiveParams) -> int:
    return int(lib().tahq_qnaive_workspace_bound(C.byref(p.c())))


def tahq_qnaive_encode(p: QNaiveParams, d_in: int, d_packed: int, cap: int, d_ws: int, ws_cap: int, stream: int) -> int:
    return (_call or call()).qnaive_encode(p.raw(), d_in, d_packed, cap, d_ws, ws_cap, stream)


def tahq_qnaive_decode(p: QNaiveParams, d_packed: int, nbytes: int, d_out: int, d_ws: int, ws_cap: int, stream: int) -> int:
    return (_call or call()).qnaive_decode(p.raw(), d_packed, nbytes, d_out, d_ws, ws_cap, stream)


def _stream_of(t: torch.Tensor) -> int:
    """The current stream of the tensor's device.  A tensor that is not on a GPU has none: the kernels could not reach it."""
    device = t.get_device()
    if device < 0:
        raise ValueError(f"Expected a cuda device, but got: {t.device}")
    return _raw_stream(device)


def qnaive_encode(p: QNaiveParams, x: torch.Tensor, packed: torch.Tensor | None = None, ws: torch.Tensor | None = None):
    if packed is None:
        packed = torch.empty(qnaive_packed_bound(p), dtype=torch.uint8, device=x.device)
    if ws is None:
        ws = torch.empty(qnaive_workspace_bound(p), dtype=torch.uint8, device=x.device)
    rc = (_call or call()).qnaive_encode(p._box[0] or p.raw(), x.data_ptr(), packed.data_ptr(), packed.numel(), ws.data_ptr(),
                                         ws.numel(), _stream_of(x))
    if rc:
        raise TahqError(rc)
    return packed, ws


def qnaive_decode(p: QNaiveParams, packed: torch.Tensor, out: torch.Tensor | None = None, ws: torch.Tensor | None = None):
    if out is None:
        out = torch.empty((p.tokens, p.hidden), device=packed.device,
                          dtype=torch.float32 if p.dtype == F32 else torch.bfloat16)
    if ws is None:
        ws = torch.empty(qnaive_workspace_bound(p), dtype=torch.uint8, device=packed.device)
    rc = (_call or call()).qnaive_decode(p._box[0] or p.raw(), packed.data_ptr(), packed.numel(), out.data_ptr(), ws.data_ptr(),
                                         ws.numel(), _stream_of(packed))
    if rc:
        raise TahqError(rc)
    return out, ws


def selftest_wait_timeout(ws: torch.Tensor) -> int:
    """Run the bounded-wait self-test on `ws` (>= 32 KiB, device); returns the C status code."""
    return int(lib().tahq_selftest_wait_timeout(ws.data_ptr(), ws.numel(), int(torch.cuda.current_stream(ws.device).cuda_stream)))
