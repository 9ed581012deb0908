"""Thin binding over libkata.so (argument marshalling only; every step runs in the CUDA
library).  Function names mirror the C ABI of include/kata.h.  The ordinary tensor call goes through a native module
(csrc/kata_torch.cpp), every other one, and every error, through ctypes here.

Tensors are torch CUDA tensors (or pinned host tensors for ``kata_fwd_host``); torch is used for
device memory and streams only.  There is no CPU fallback: if the library is missing or a call
fails, an exception is raised.
"""
from __future__ import annotations

import collections
import ctypes
import functools
import os
import threading
import warnings
from typing import Optional

import torch

from . import build

HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(HERE, "libkata.so")

KATA_F32, KATA_BF16 = 0, 1
KATA_LAYOUT_DIRECT, KATA_LAYOUT_PACKED = 0, 1
KATA_SEQUENTIAL, KATA_SCAN, KATA_INTER_AUTO = 0, 1, 2
KATA_IMPL_AUTO, KATA_IMPL_SIMT, KATA_IMPL_TENSOR = 0, 1, 2
KATA_FN_QUADRATIC, KATA_FN_CHUNKED, KATA_FN_CHUNK_STATE_SCAN, KATA_FN_DECODE_STEP = 0, 1, 2, 3
KATA_FN_BWD_QUADRATIC = 4
KATA_FN_BWD_CHUNKED = 5
KATA_FN_HOST_IO = 0x100
KATA_OK, KATA_ERR_INVALID_ARG, KATA_ERR_UNSUPPORTED_SHAPE, KATA_ERR_WORKSPACE_TOO_SMALL, KATA_ERR_DEVICE_TIMEOUT = 0, -1, -2, -4, -7

EXPORTS = ("kata_fwd_quadratic", "kata_fwd_chunked", "kata_chunk_state_scan", "kata_chunk_state_scan_static",
           "kata_fwd_host", "kata_decode_step", "kata_bwd_quadratic", "kata_bwd_chunked",
           "kata_workspace_bytes", "kata_scan_plan", "kata_host_plan", "kata_last_launch_count", "kata_last_impl",
           "kata_status_string",
           "kata_version")


class KataOpts(ctypes.Structure):
    _fields_ = [
        ("struct_size", ctypes.c_uint32),
        ("dtype", ctypes.c_int32),
        ("feature_order", ctypes.c_int32),
        ("state_layout", ctypes.c_int32),
        ("inter_chunk", ctypes.c_int32),
        ("impl", ctypes.c_int32),
        ("scan_group", ctypes.c_int32),
        ("feature_groups", ctypes.c_int32),
        ("workspace", ctypes.c_void_p),
        ("workspace_bytes", ctypes.c_size_t),
        ("s_pre", ctypes.c_void_p),
        ("z_pre", ctypes.c_void_p),
        ("device_status", ctypes.c_void_p),
        ("stream", ctypes.c_void_p),
        ("s_init", ctypes.c_void_p),
        ("z_init", ctypes.c_void_p),
    ]


class KataError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {status_string(status)} ({status})")


_lib = None


def lib() -> ctypes.CDLL:
    """Load libkata.so (once).  Raises if it has not been built."""
    global _lib
    if _lib is not None:
        return _lib
    if not os.path.exists(LIB_PATH):
        raise RuntimeError(f"{LIB_PATH} not found: build it with `python -m paper_2607_17419_b200.build`")
    L = ctypes.CDLL(LIB_PATH)
    ptr, i = ctypes.c_void_p, ctypes.c_int
    fwd_args = [ptr, ptr, ptr, ptr, i, i, i, i, i, i, ctypes.POINTER(KataOpts)]
    for name in ("kata_fwd_quadratic", "kata_fwd_chunked", "kata_chunk_state_scan", "kata_chunk_state_scan_static"):
        getattr(L, name).argtypes = fwd_args
        getattr(L, name).restype = i
    L.kata_fwd_host.argtypes = [i] + fwd_args
    L.kata_fwd_host.restype = i
    L.kata_decode_step.argtypes = [ptr, ptr, ptr, ptr, ptr, ptr, i, i, i, i, ctypes.POINTER(KataOpts)]
    L.kata_decode_step.restype = i
    L.kata_bwd_quadratic.argtypes = [ptr] * 7 + [i] * 5 + [ctypes.POINTER(KataOpts)]
    L.kata_bwd_quadratic.restype = i
    L.kata_bwd_chunked.argtypes = [ptr] * 7 + [i] * 6 + [ctypes.POINTER(KataOpts)]
    L.kata_bwd_chunked.restype = i
    L.kata_workspace_bytes.argtypes = [i, i, i, i, i, i, i, ctypes.POINTER(KataOpts)]
    L.kata_workspace_bytes.restype = ctypes.c_size_t
    L.kata_scan_plan.argtypes = [i, i, i, i, i, i, i, ctypes.POINTER(KataOpts)] + [ctypes.POINTER(i)] * 3
    L.kata_scan_plan.restype = i
    L.kata_host_plan.argtypes = [i, i, i, i, i, i, i, ctypes.POINTER(KataOpts)] + [ctypes.POINTER(i)] * 2
    L.kata_host_plan.restype = i
    L.kata_last_launch_count.argtypes = []
    L.kata_last_launch_count.restype = i
    L.kata_last_impl.argtypes = []
    L.kata_last_impl.restype = i
    L.kata_status_string.argtypes = [i]
    L.kata_status_string.restype = ctypes.c_char_p
    L.kata_version.argtypes = []
    L.kata_version.restype = i
    L.kata_selftest_wait_timeout.argtypes = [ptr, ptr, ctypes.c_uint, ptr]
    L.kata_selftest_wait_timeout.restype = i
    _lib = L
    return L


_native = None


class _CtypesOnly:
    """In the native module's place where it cannot be used: every call is left to this file."""

    @staticmethod
    def forward(*args):
        return NotImplemented

    decode = backward = forward


def native():
    """The native module with the tensor calls (loaded once); each returns NotImplemented for a call that is left to this file.
    Where the module is missing, does not load or was built for another torch or Python, all calls are, with one warning."""
    global _native
    if _native is None:
        lib()
        why = None
        if build.host_current():
            try:
                from . import _kata_torch
                _native = _kata_torch
            except ImportError as e:
                why = f"does not load ({e})"
        elif os.path.exists(build.HOST):
            why = "was built for another torch or Python"
        else:
            why = "is missing"
        if why is not None:
            warnings.warn(f"_kata_torch.so {why}: calls take some 5 us more on the host; `python -m paper_2607_17419_b200.build` builds it")
            _native = _CtypesOnly
    return _native


def status_string(status: int) -> str:
    return lib().kata_status_string(status).decode()


_OPTS_SIZE = ctypes.sizeof(KataOpts)


def make_opts(dtype: int, *, feature_order: int = 2, state_layout: int = KATA_LAYOUT_DIRECT,
              inter_chunk: int = KATA_SEQUENTIAL, impl: int = KATA_IMPL_AUTO, scan_group: int = 0,
              feature_groups: int = 0,
              workspace: int = 0, workspace_bytes: int = 0, s_pre: int = 0, z_pre: int = 0,
              device_status: int = 0, stream: int = 0, s_init: int = 0, z_init: int = 0) -> KataOpts:
    # (one constructor call: setting the fields one by one costs 3 us of a 10 us call)
    return KataOpts(_OPTS_SIZE, dtype, feature_order, state_layout, inter_chunk, impl, scan_group, feature_groups,
                    workspace or None, workspace_bytes, s_pre or None, z_pre or None, device_status or None, stream or None,
                    s_init or None, z_init or None)


def kata_workspace_bytes(fn: int, B, H, T, d_k, d_v, C, opts: KataOpts) -> int:
    return int(lib().kata_workspace_bytes(fn, B, H, T, d_k, d_v, C, ctypes.byref(opts)))


@functools.lru_cache(maxsize=4096)
def _scratch_bytes(fn: int, B, H, T, d_k, d_v, C, dtype, order, layout, inter, impl, scan_group, groups, state_in: bool,
                   state_out: bool, in_place: bool) -> int:
    """kata_workspace_bytes as what it is: a function of the sizes, the options and which state pointers are set."""
    o = make_opts(dtype, feature_order=order, state_layout=layout, inter_chunk=inter, impl=impl, scan_group=scan_group,
                  feature_groups=groups, s_pre=256 if state_out else 0, z_pre=256 if state_out else 0,
                  s_init=(256 if in_place else 512) if state_in else 0, z_init=(256 if in_place else 512) if state_in else 0)
    return kata_workspace_bytes(fn, B, H, T, d_k, d_v, C, o)


def _scratch(ws, fn: int, sizes, o: KataOpts, device):
    """Point the options at scratch of the size the call needs; the caller holds what is returned until the call is made."""
    need = _scratch_bytes(fn, *sizes, o.dtype, o.feature_order, o.state_layout, o.inter_chunk, o.impl, o.scan_group,
                          o.feature_groups, bool(o.s_init or o.z_init), bool(o.s_pre or o.z_pre),
                          o.z_init is not None and o.z_init == o.z_pre)
    if ws is not None:
        ptr, size = ws.get(need, device)
        if size:
            o.workspace, o.workspace_bytes = ptr, size
        return ws
    if need == 0:
        return None
    stream = o.stream                   # (None: the legacy default stream, which cannot be captured)
    held = _default_scratch.bufs.get((device.index, stream))
    if held is None or held[2] < need or (stream is not None and torch._C._cuda_isCurrentStreamCapturing()):
        held = _default_scratch.new(need, device, stream)
    o.workspace, o.workspace_bytes = held[1], held[2]
    return held


def kata_scan_plan(fn: int, B, H, T, d_k, d_v, C, opts: KataOpts):
    """(n_groups, chunks_per_group, scan_rounds) the library would use."""
    a, b, c = ctypes.c_int(), ctypes.c_int(), ctypes.c_int()
    st = lib().kata_scan_plan(fn, B, H, T, d_k, d_v, C, ctypes.byref(opts), ctypes.byref(a), ctypes.byref(b),
                              ctypes.byref(c))
    if st != 0:
        raise KataError(st, "kata_scan_plan")
    return a.value, b.value, c.value


def kata_host_plan(fn: int, B, H, T, d_k, d_v, C, opts: KataOpts):
    """(pieces, tokens per piece) the host-buffer entry would work in."""
    a, b = ctypes.c_int(), ctypes.c_int()
    st = lib().kata_host_plan(fn, B, H, T, d_k, d_v, C, ctypes.byref(opts), ctypes.byref(a), ctypes.byref(b))
    if st != 0:
        raise KataError(st, "kata_host_plan")
    return a.value, b.value


def kata_selftest_wait_timeout(device_status, report, max_polls: int = 1000, stream=None) -> int:
    """Test hook (csrc/kata_selftest.h): one warp runs both bounded waits on a barrier nobody arrives at.

    `device_status` is an int32 CUDA tensor of one element (or None), `report` one of eight (the last is the flag in
    global memory that the flag wait is tried on: 0 on entry).  Returns the status code.
    """
    if stream is None:
        stream = torch.cuda.current_stream().cuda_stream
    return int(lib().kata_selftest_wait_timeout(device_status.data_ptr() if device_status is not None else None,
                                                report.data_ptr() if report is not None else None, max_polls, stream))


def kata_last_launch_count() -> int:
    return int(lib().kata_last_launch_count())


def kata_last_impl() -> int:
    return int(lib().kata_last_impl())


def kata_version() -> int:
    return int(lib().kata_version())


# ---------------------------------------------------------------------------
# tensor-level wrappers
# ---------------------------------------------------------------------------

_FN_NAMES = {KATA_FN_QUADRATIC: "kata_fwd_quadratic", KATA_FN_CHUNKED: "kata_fwd_chunked",
             KATA_FN_CHUNK_STATE_SCAN: "kata_chunk_state_scan"}


_DTYPE_CODES = {torch.float32: KATA_F32, torch.bfloat16: KATA_BF16}


def _dtype_code(t) -> int:
    try:
        return _DTYPE_CODES[t.dtype]
    except KeyError:
        raise TypeError(f"unsupported dtype {t.dtype}") from None


def _stream(device) -> int:
    """Handle of torch's current stream on the device (without the stream object: 2 us of a 10 us call)."""
    return torch._C._cuda_getCurrentRawStream(device.index)


class Workspace:
    """A reusable device scratch buffer (torch allocation, grown on demand)."""

    def __init__(self):
        self.buf = None

    def get(self, nbytes: int, device):
        if nbytes == 0:
            return 0, 0
        buf = self.buf
        if buf is None or buf.numel() < nbytes or buf.device != device:
            self.buf = buf = torch.empty(nbytes, dtype=torch.uint8, device=device)
        return buf.data_ptr(), buf.numel()


class _StreamScratch(threading.local):
    """Scratch of the calls that bring no Workspace: a buffer per thread, device and stream, so that calls on different
    streams or threads never share one.  The buffers belong to their streams in torch's allocator (one that is replaced is
    used again behind the calls that still read it), the oldest of more than KEEP goes back to it, and all of a thread's go
    with the thread.  A call under graph capture gets a buffer of its own from the graph's pool (a capture that torch did not
    begin has no pool: bring a Workspace)."""

    KEEP = 16

    def __init__(self):
        self.bufs = {}                  # (device index, stream) -> (buffer, its address, its size)

    def new(self, nbytes: int, device, stream: Optional[int]):
        if (stream or 0) == _stream(device):
            buf = torch.empty(nbytes, dtype=torch.uint8, device=device)
        else:
            with torch.cuda.stream(torch.cuda.ExternalStream(stream or 0, device=device)):
                buf = torch.empty(nbytes, dtype=torch.uint8, device=device)
        held = (buf, buf.data_ptr(), nbytes)
        if not torch.cuda.is_current_stream_capturing():
            self.bufs.pop((device.index, stream), None)
            self.bufs[device.index, stream] = held
            if len(self.bufs) > self.KEEP:
                del self.bufs[next(iter(self.bufs))]
        return held


_default_scratch = _StreamScratch()


def _on(t, device) -> bool:
    """Whether kernels on the device can address the tensor."""
    return t.device == device or (t.device.type == "cpu" and t.is_pinned())


def _check_room(q, heads: int, inputs, outputs, state=(), host_io: bool = False):
    """ValueError for a tensor that the kernels, which take sizes, type and device from q (and d_v from v), would read or write
    beyond its end or misread.  Each group holds (name, tensor or None, elements that the call touches).  Inputs have that many
    elements, in any shape; with one head, where nothing lies behind them, they may have more, as outputs and state may.
    (The native module, given no scratch, looks first in 0.1 us: this takes 3 to 6, a third of a small call.)"""
    for group, dtype in ((inputs, q.dtype), (outputs, q.dtype), (state, torch.float32)):
        for name, t, n in group:
            if not isinstance(t, torch.Tensor):
                continue
            size = t.numel()
            if size != n and (size < n or (group is inputs and heads > 1)):
                raise ValueError(f"{name} has {size} elements, the call needs {n}")
            if t.dtype is not dtype:
                raise ValueError(f"{name} is {t.dtype}, the call needs {dtype}")
            if not host_io and not _on(t, q.device):
                raise ValueError(f"{name} is on {t.device}, q on {q.device}")
            if not t.is_contiguous():
                raise ValueError(f"{name} must be contiguous")


def _check_forward(fn: int, q, k, v, out, C, host_io=False, s_pre=None, z_pre=None, s_init=None, z_init=None, device_status=None,
                   feature_order=2, state_layout=KATA_LAYOUT_DIRECT, feature_groups=0, **_):
    B, H, T, d_k = q.shape
    d_v, heads = v.shape[-1], B * H
    state = ()
    if s_pre is not None or z_pre is not None or s_init is not None or z_init is not None:
        rows = heads * decode_n_psi(d_k, feature_order, state_layout, feature_groups)
        rows_pre = rows * -(-T // C) if fn == KATA_FN_CHUNK_STATE_SCAN and C > 0 else rows
        state = (("s_pre", s_pre, rows_pre * d_v), ("z_pre", z_pre, rows_pre), ("s_init", s_init, rows * d_v), ("z_init", z_init, rows))
    _check_room(q, heads, (("k", k, heads * T * d_k), ("v", v, heads * T * d_v)), (("out", out, heads * T * d_v),), state, host_io)
    if isinstance(device_status, torch.Tensor) and (device_status.nbytes < 4 or not (host_io or _on(device_status, q.device))):
        raise ValueError("device_status is one int32 on the device of q")


def _check_backward(q, k, v, dout, dq, dk, dv):
    B, H, T, d_k = q.shape
    nk, nv = B * H * T * d_k, B * H * T * v.shape[-1]
    _check_room(q, B * H, (("k", k, nk), ("v", v, nv), ("dout", dout, nv)), (("dq", dq, nk), ("dk", dk, nk), ("dv", dv, nv)))


def _call(fn: int, q, k, v, out, C: int, *, host_io: bool = False, workspace: Optional[Workspace] = None,
          s_pre=None, z_pre=None, s_init=None, z_init=None, device_status=None, stream=None, **opt_kw):
    if workspace is None and stream is None and not host_io:
        r = (_native or native()).forward(fn, _default_scratch, q, k, v, out, C, s_pre, z_pre, s_init, z_init, device_status, opt_kw)
        if type(r) is int:
            raise KataError(r, _FN_NAMES[fn])
        if r is not NotImplemented:
            return r
    if not (q.is_contiguous() and k.is_contiguous() and v.is_contiguous()):
        raise ValueError("q, k, v must be contiguous [B,H,T,d]")
    B, H, T, d_k = q.shape
    d_v = v.shape[-1]
    if host_io or (_native or native()).forward(fn, None, q, k, v, out, C, s_pre, z_pre, s_init, z_init, device_status, opt_kw) is not True:
        _check_forward(fn, q, k, v, out, C, host_io, s_pre, z_pre, s_init, z_init, device_status, **opt_kw)
    if out is None:
        out = torch.empty_like(v)
    dev = torch.device("cuda", torch.cuda.current_device()) if host_io else q.device
    if stream is None:
        stream = _stream(dev)
    opts = make_opts(_dtype_code(q), stream=stream,
                     s_pre=s_pre.data_ptr() if s_pre is not None else 0,
                     z_pre=z_pre.data_ptr() if z_pre is not None else 0,
                     s_init=s_init.data_ptr() if s_init is not None else 0,
                     z_init=z_init.data_ptr() if z_init is not None else 0,
                     device_status=device_status.data_ptr() if device_status is not None else 0, **opt_kw)
    held = _scratch(workspace, fn | (KATA_FN_HOST_IO if host_io else 0), (B, H, T, d_k, d_v, C), opts, dev)
    args = (q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), B, H, T, d_k, d_v, C, ctypes.byref(opts))
    if host_io:
        st = lib().kata_fwd_host(fn, *args)
        name = "kata_fwd_host"
    else:
        name = _FN_NAMES[fn]
        st = getattr(lib(), name)(*args)
    if st != 0:
        raise KataError(st, name)
    return out


def kata_fwd_quadratic(q, k, v, out=None, C: int = 64, **kw):
    """Quadratic forward; q,k [B,H,T,d_k], v [B,H,T,d_v] CUDA tensors (fp32 or bf16)."""
    return _call(KATA_FN_QUADRATIC, q, k, v, out, C, **kw)


def kata_fwd_chunked(q, k, v, out=None, C: int = 64, **kw):
    """Chunked-state forward; inter_chunk=KATA_SEQUENTIAL (default), KATA_SCAN or KATA_INTER_AUTO.  In the sequential form
    s_init/z_init give the state before the first token and s_pre/z_pre receive the state after the last."""
    return _call(KATA_FN_CHUNKED, q, k, v, out, C, **kw)


def kata_chunk_state_scan(q, k, v, out=None, C: int = 64, **kw):
    """Chunk-state -> log-depth scan -> chunk-output pipeline; optional s_pre/z_pre export."""
    return _call(KATA_FN_CHUNK_STATE_SCAN, q, k, v, out, C, **kw)


def kata_fwd_host(fn: int, q, k, v, out, C: int = 64, **kw):
    """Same as entry point ``fn`` with (pinned) host tensors; copies ride the current CUDA stream."""
    return _call(fn, q, k, v, out, C, host_io=True, **kw)


def decode_n_psi(d_k: int, feature_order: int = 2, state_layout: int = KATA_LAYOUT_DIRECT, feature_groups: int = 0) -> int:
    """Feature rows of the state: d_k (order 1); g m^2 (direct) or g m(m+1)/2 (packed) with m = d_k / g for the
    PSD lift in g blocks (g = 1: the full lift)."""
    if feature_order == 1:
        return d_k
    g = max(1, feature_groups)
    m = d_k // g
    return g * (m * (m + 1) // 2 if state_layout == KATA_LAYOUT_PACKED else m * m)


def kata_decode_step(q, k, v, S, Z, out=None, *, workspace: Optional[Workspace] = None, stream=None, **opt_kw):
    """One decode token per (b,h): q,k [B,H,d_k], v [B,H,d_v]; fp32 state S [B,H,n_psi,d_v], Z [B,H,n_psi] is
    updated in place.  Returns out [B,H,d_v]."""
    if workspace is None and stream is None:
        r = (_native or native()).decode(_default_scratch, q, k, v, S, Z, out, opt_kw)
        if type(r) is int:
            raise KataError(r, "kata_decode_step")
        if r is not NotImplemented:
            return r
    B, H, d_k = q.shape
    d_v = v.shape[-1]
    if not (q.is_contiguous() and k.is_contiguous() and v.is_contiguous() and S.is_contiguous() and Z.is_contiguous()):
        raise ValueError("q, k, v, S, Z must be contiguous")
    if S.dtype != torch.float32 or Z.dtype != torch.float32:
        raise ValueError("the state is fp32")
    if (_native or native()).decode(None, q, k, v, S, Z, out, opt_kw) is not True:
        _check_room(q, B * H, (("k", k, B * H * d_k), ("v", v, B * H * d_v)), (("out", out, B * H * d_v),),
                    (("S", S, 0), ("Z", Z, 0)))               # (the sizes of the state: below)
    if out is None:
        out = torch.empty_like(v)
    if stream is None:
        stream = _stream(q.device)
    opts = make_opts(_dtype_code(q), stream=stream, **opt_kw)
    n_psi = decode_n_psi(d_k, opts.feature_order, opts.state_layout, opts.feature_groups)
    if S.shape != (B, H, n_psi, d_v) or Z.shape != (B, H, n_psi):
        raise ValueError(f"state shapes must be {(B, H, n_psi, d_v)} and {(B, H, n_psi)}")
    held = _scratch(workspace, KATA_FN_DECODE_STEP, (B, H, 1, d_k, d_v, 0), opts, q.device)
    st = lib().kata_decode_step(q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), S.data_ptr(), Z.data_ptr(),
                                B, H, d_k, d_v, ctypes.byref(opts))
    if st != 0:
        raise KataError(st, "kata_decode_step")
    return out


def kata_bwd_quadratic(q, k, v, dout, dq=None, dk=None, dv=None, *, workspace: Optional[Workspace] = None,
                       stream=None, **opt_kw):
    """Gradients of sum(dout * out) with respect to q, k, v (q,k [B,H,T,d_k]; v,dout [B,H,T,d_v]); the forward
    is recomputed.  Returns (dq, dk, dv) in the dtype of the inputs."""
    if workspace is None and stream is None:
        r = (_native or native()).backward(KATA_FN_BWD_QUADRATIC, _default_scratch, q, k, v, dout, dq, dk, dv, 0, opt_kw)
        if type(r) is int:
            raise KataError(r, "kata_bwd_quadratic")
        if r is not NotImplemented:
            return r
    if not (q.is_contiguous() and k.is_contiguous() and v.is_contiguous() and dout.is_contiguous()):
        raise ValueError("q, k, v, dout must be contiguous [B,H,T,d]")
    B, H, T, d_k = q.shape
    d_v = v.shape[-1]
    if (_native or native()).backward(KATA_FN_BWD_QUADRATIC, None, q, k, v, dout, dq, dk, dv, 0, opt_kw) is not True:
        _check_backward(q, k, v, dout, dq, dk, dv)
    dq = torch.empty_like(q) if dq is None else dq
    dk = torch.empty_like(k) if dk is None else dk
    dv = torch.empty_like(v) if dv is None else dv
    if stream is None:
        stream = _stream(q.device)
    opts = make_opts(_dtype_code(q), stream=stream, **opt_kw)
    held = _scratch(workspace, KATA_FN_BWD_QUADRATIC, (B, H, T, d_k, d_v, 0), opts, q.device)
    st = lib().kata_bwd_quadratic(q.data_ptr(), k.data_ptr(), v.data_ptr(), dout.data_ptr(), dq.data_ptr(),
                                  dk.data_ptr(), dv.data_ptr(), B, H, T, d_k, d_v, ctypes.byref(opts))
    if st != 0:
        raise KataError(st, "kata_bwd_quadratic")
    return dq, dk, dv


def kata_bwd_chunked(q, k, v, dout, dq=None, dk=None, dv=None, C: int = 64, *, workspace: Optional[Workspace] = None,
                     stream=None, **opt_kw):
    """The same gradients as ``kata_bwd_quadratic`` by the O(T) two-pass linear-state backward.  Returns (dq, dk, dv)
    in the dtype of the inputs."""
    if workspace is None and stream is None:
        r = (_native or native()).backward(KATA_FN_BWD_CHUNKED, _default_scratch, q, k, v, dout, dq, dk, dv, C, opt_kw)
        if type(r) is int:
            raise KataError(r, "kata_bwd_chunked")
        if r is not NotImplemented:
            return r
    if not (q.is_contiguous() and k.is_contiguous() and v.is_contiguous() and dout.is_contiguous()):
        raise ValueError("q, k, v, dout must be contiguous [B,H,T,d]")
    B, H, T, d_k = q.shape
    d_v = v.shape[-1]
    if (_native or native()).backward(KATA_FN_BWD_CHUNKED, None, q, k, v, dout, dq, dk, dv, C, opt_kw) is not True:
        _check_backward(q, k, v, dout, dq, dk, dv)
    dq = torch.empty_like(q) if dq is None else dq
    dk = torch.empty_like(k) if dk is None else dk
    dv = torch.empty_like(v) if dv is None else dv
    if stream is None:
        stream = _stream(q.device)
    opts = make_opts(_dtype_code(q), stream=stream, **opt_kw)
    held = _scratch(workspace, KATA_FN_BWD_CHUNKED, (B, H, T, d_k, d_v, C), opts, q.device)
    st = lib().kata_bwd_chunked(q.data_ptr(), k.data_ptr(), v.data_ptr(), dout.data_ptr(), dq.data_ptr(),
                                dk.data_ptr(), dv.data_ptr(), B, H, T, d_k, d_v, C, ctypes.byref(opts))
    if st != 0:
        raise KataError(st, "kata_bwd_chunked")
    return dq, dk, dv


KATA_STATIC_SCRATCH_BYTES = 32 << 20


def kata_chunk_state_scan_static(q, k, v, out, C: int = 64, *, scan_group: int = 0, impl: int = KATA_IMPL_AUTO,
                                 feature_order: int = 2, stream=None):
    """The scan pipeline with the library's built-in scratch: for callers that must not allocate.

    Unlike the other wrappers this one never touches torch's allocator: ``out`` must be passed in, and
    no workspace is requested.  Calls that overlap on the GPU share (and race on) the one scratch array.
    """
    B, H, T, d_k = q.shape
    d_v = v.shape[-1]
    if not (q.is_contiguous() and k.is_contiguous() and v.is_contiguous()):
        raise ValueError("q, k, v must be contiguous [B,H,T,d]")
    if (_native or native()).forward(KATA_FN_CHUNK_STATE_SCAN, None, q, k, v, out, C, None, None, None, None, None, {}) is not True:
        _check_forward(KATA_FN_CHUNK_STATE_SCAN, q, k, v, out, C)
    if stream is None:
        stream = _stream(q.device)
    opts = make_opts(_dtype_code(q), stream=stream, scan_group=scan_group, impl=impl, feature_order=feature_order)
    st = lib().kata_chunk_state_scan_static(q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), B, H, T, d_k, d_v,
                                            C, ctypes.byref(opts))
    if st != 0:
        raise KataError(st, "kata_chunk_state_scan_static")
    return out
