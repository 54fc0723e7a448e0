"""Binding of libhola_verify.so (ctypes, and native code for the calls of a serving loop, csrc/host_call.cpp): argument
marshalling only, every step runs in the CUDA kernels.

Function names mirror the C ABI (include/hola_verify.h).  Tensors are torch CUDA tensors; torch is used for
device memory and streams, nothing else.
"""
from __future__ import annotations

import ctypes
import os
import subprocess
import warnings
from array import array
from dataclasses import dataclass

import torch

from . import build as _build

HOLA_OK = 0
HOLA_Q_BF16, HOLA_Q_F32 = 0, 1
HOLA_GATE_TARGET_ENTROPY, HOLA_GATE_DRAFT_ENTROPY = 0, 1
HOLA_FALLBACK_SAMPLE, HOLA_FALLBACK_GREEDY = 0, 1
HOLA_W_BF16, HOLA_W_INT8, HOLA_W8A8, HOLA_W8A16, HOLA_W_MIXED = 0, 1, 2, 3, 4
HOLA_HIDDEN_IN_PLACE, HOLA_HIDDEN_ON_LINES, HOLA_HIDDEN_8BIT = 0, 1, 2
HOLA_ARG_CLEAR_STATUS = 1
GROUP_ROWS, SUB_BLOCK, HOLA_PACE_WORDS = 256, 128, 256
FLAG_BAD_TOKEN, FLAG_BAD_UNIFORM, FLAG_TIMEOUT, FLAG_R_ZERO = 1, 2, 4, 8
HOLA_OPT_RING_SLOTS, HOLA_OPT_ROTATING_UNITS, HOLA_OPT_HOST_OVERLAP, HOLA_OPT_HOST_ROWS_ON_DEMAND, HOLA_OPT_PASSES, HOLA_OPT_PAIR_MMA, HOLA_OPT_HOST_IN_PLACE, HOLA_OPT_CONVERTER_GROUP, HOLA_OPT_FUSED_PASSES = 1, 2, 3, 4, 5, 6, 7, 8, 9

EXPORTS = ["hola_create", "hola_destroy", "hola_workspace_bytes", "hola_verify", "hola_verify_host",
           "hola_lm_head_entropy", "hola_accept_sample", "hola_host_traffic", "hola_shard_record_bytes", "hola_shard_lm_head",
           "hola_shard_accept", "hola_shard_sample", "hola_lm_head_entropy_static", "hola_quantize_w8", "hola_quantize_w4", "hola_quantize_mixed", "hola_quantize_mixed_widths", "hola_plan", "hola_plan_ex", "hola_plan_for_shape", "hola_hidden_form_for_shape", "hola_sample_plan_for_shape", "hola_set_option", "hola_selftest_bounded_wait", "hola_selftest_staged_wait", "hola_selftest_mass_wait", "hola_selftest_pace", "hola_selftest_quotient", "hola_profile_begin", "hola_profile_end", "hola_strerror", "hola_last_cuda_error",
           "hola_version"]


class HolaError(RuntimeError):
    pass


class hola_verify_args(ctypes.Structure):
    _fields_ = [("B", ctypes.c_int32), ("k", ctypes.c_int32), ("H", ctypes.c_int32), ("V", ctypes.c_int32),
                ("hidden", ctypes.c_void_p), ("W_lm", ctypes.c_void_p), ("draft_tok", ctypes.c_void_p),
                ("draft_q", ctypes.c_void_p), ("q_dtype", ctypes.c_int32), ("uniforms", ctypes.c_void_p),
                ("tau", ctypes.c_float), ("accept_len", ctypes.c_void_p), ("next_tok", ctypes.c_void_p),
                ("entropy", ctypes.c_void_p), ("logZ", ctypes.c_void_p), ("logits_out", ctypes.c_void_p),
                ("status_word", ctypes.c_void_p), ("gate_source", ctypes.c_int32), ("fallback", ctypes.c_int32),
                ("draft_entropy", ctypes.c_void_p), ("w_dtype", ctypes.c_int32), ("flags", ctypes.c_int32),
                ("w_scale", ctypes.c_void_p), ("wmix", ctypes.c_void_p)]


class hola_wmix(ctypes.Structure):
    _fields_ = [("W16", ctypes.c_void_p), ("W8", ctypes.c_void_p), ("W4", ctypes.c_void_p), ("shift4", ctypes.c_void_p),
                ("group_width", ctypes.c_void_p), ("group_row", ctypes.c_void_p), ("rows16", ctypes.c_int32),
                ("rows8", ctypes.c_int32), ("rows4", ctypes.c_int32), ("reserved_", ctypes.c_int32)]


class hola_shard_args(ctypes.Structure):
    _fields_ = [("world", ctypes.c_int32), ("rank", ctypes.c_int32), ("v_offset", ctypes.c_int32),
                ("V_global", ctypes.c_int32), ("q_tok", ctypes.c_void_p), ("record_out", ctypes.c_void_p),
                ("records", ctypes.c_void_p), ("mass_out", ctypes.c_void_p), ("masses", ctypes.c_void_p)]


class hola_plan_info(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in ("tile_v", "grid", "stages", "rows_per_pass", "passes", "kernels_per_call")]


class hola_sample_info(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in ("ctas", "threads", "staged")]


_lib = None
_host = None            # the native helper (csrc/host_call.cpp), or None: arguments are then filled from Python
_entry = {}             # addresses of the entry points that it calls


def _load_host(lib: ctypes.CDLL):
    """The helper reads tensors through torch's C++ classes: it is built against the torch that runs."""
    global _host
    try:
        helper = _build.load_host()
    except (ImportError, OSError, subprocess.CalledProcessError) as e:
        warnings.warn(f"host-side helper not available, calls cost a few microseconds more: {e}")
        return
    for name in ("hola_verify", "hola_verify_host", "hola_lm_head_entropy", "hola_quantize_mixed_widths"):
        _entry[name] = ctypes.cast(getattr(lib, name), ctypes.c_void_p).value
    _host = helper


def load_library(path: str | None = None) -> ctypes.CDLL:
    """Loads the C-ABI library (building it first if the source is newer).  Raises if it cannot be had."""
    global _lib
    if _lib is not None and path is None:
        return _lib
    p = path or (_build.LIB if os.path.exists(_build.LIB) and not _build.needs_build() else _build.build())
    lib = ctypes.CDLL(p)
    lib.hola_create.restype = ctypes.c_int
    lib.hola_create.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_int, ctypes.c_int, ctypes.c_int,
                                ctypes.c_int, ctypes.c_int]
    lib.hola_destroy.restype = ctypes.c_int
    lib.hola_destroy.argtypes = [ctypes.c_void_p]
    lib.hola_workspace_bytes.restype = ctypes.c_size_t
    lib.hola_workspace_bytes.argtypes = [ctypes.c_int] * 4
    for name in ("hola_verify", "hola_verify_host", "hola_lm_head_entropy", "hola_accept_sample"):
        fn = getattr(lib, name)
        fn.restype = ctypes.c_int
        fn.argtypes = [ctypes.c_void_p, ctypes.POINTER(hola_verify_args), ctypes.c_void_p]
    lib.hola_lm_head_entropy_static.restype = ctypes.c_int
    lib.hola_lm_head_entropy_static.argtypes = [ctypes.POINTER(hola_verify_args), ctypes.c_void_p]
    lib.hola_quantize_w8.restype = ctypes.c_int
    lib.hola_quantize_w8.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p,
                                     ctypes.c_void_p]
    lib.hola_quantize_w4.restype = ctypes.c_int
    lib.hola_quantize_w4.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p,
                                     ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    lib.hola_quantize_mixed.restype = ctypes.c_int
    lib.hola_quantize_mixed.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.POINTER(hola_wmix),
                                        ctypes.c_void_p, ctypes.c_void_p]
    lib.hola_quantize_mixed_widths.restype = ctypes.c_int
    lib.hola_quantize_mixed_widths.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p,
                                               ctypes.POINTER(hola_wmix), ctypes.c_void_p, ctypes.c_void_p]
    lib.hola_plan.restype = ctypes.c_int
    lib.hola_plan.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.POINTER(hola_plan_info)]
    lib.hola_plan_for_shape.restype = ctypes.c_int
    lib.hola_plan_for_shape.argtypes = [ctypes.c_int] * 5 + [ctypes.POINTER(hola_plan_info)]
    lib.hola_hidden_form_for_shape.restype = ctypes.c_int
    lib.hola_hidden_form_for_shape.argtypes = [ctypes.c_int] * 5 + [ctypes.POINTER(ctypes.c_int32)]
    lib.hola_sample_plan_for_shape.restype = ctypes.c_int
    lib.hola_sample_plan_for_shape.argtypes = [ctypes.c_int] * 6 + [ctypes.POINTER(hola_sample_info)]
    lib.hola_plan_ex.restype = ctypes.c_int
    lib.hola_plan_ex.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.POINTER(hola_plan_info)]
    lib.hola_profile_begin.restype = ctypes.c_int
    lib.hola_profile_begin.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.hola_set_option.restype = ctypes.c_int
    lib.hola_set_option.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    for name in ("hola_selftest_bounded_wait", "hola_selftest_staged_wait", "hola_selftest_mass_wait"):
        fn = getattr(lib, name)
        fn.restype = ctypes.c_int
        fn.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    lib.hola_selftest_pace.restype = ctypes.c_int
    lib.hola_selftest_pace.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    lib.hola_selftest_quotient.restype = ctypes.c_int
    lib.hola_selftest_quotient.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p,
                                           ctypes.c_void_p]
    lib.hola_shard_record_bytes.restype = ctypes.c_size_t
    lib.hola_shard_record_bytes.argtypes = [ctypes.c_int, ctypes.c_int]
    for name in ("hola_shard_lm_head", "hola_shard_accept", "hola_shard_sample"):
        fn = getattr(lib, name)
        fn.restype = ctypes.c_int
        fn.argtypes = [ctypes.c_void_p, ctypes.POINTER(hola_verify_args), ctypes.POINTER(hola_shard_args),
                       ctypes.c_void_p]
    lib.hola_host_traffic.restype = ctypes.c_int
    lib.hola_host_traffic.argtypes = [ctypes.c_void_p, ctypes.POINTER(ctypes.c_ulonglong),
                                      ctypes.POINTER(ctypes.c_ulonglong)]
    lib.hola_profile_end.restype = ctypes.c_int
    lib.hola_profile_end.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.POINTER(ctypes.c_double),
                                     ctypes.POINTER(ctypes.c_double), ctypes.POINTER(ctypes.c_int)]
    lib.hola_strerror.restype = ctypes.c_char_p
    lib.hola_strerror.argtypes = [ctypes.c_int]
    lib.hola_last_cuda_error.restype = ctypes.c_char_p
    lib.hola_last_cuda_error.argtypes = [ctypes.c_void_p]
    lib.hola_version.restype = ctypes.c_char_p
    if path is None:
        _lib = lib
        _load_host(lib)
    return lib


def _check(lib, ctx, status: int, what: str):
    if status != HOLA_OK:
        msg = lib.hola_strerror(status).decode()
        detail = lib.hola_last_cuda_error(ctx).decode() if ctx else ""
        raise HolaError(f"{what}: {msg}" + (f" [{detail}]" if detail else ""))


def _dptr(t: torch.Tensor | None):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _stream_ptr(stream) -> int:
    """cudaStream_t of a torch stream; None: the current stream of the current device, without making a Stream object
    for it (a quarter of what a call costs on the host)."""
    return torch._C._cuda_getCurrentRawStream(torch._C._cuda_getDevice()) if stream is None else stream.cuda_stream


def hola_quantize_w8(W_lm: torch.Tensor, stream=None):
    """8-bit form of a bf16 W_lm [V, H] on the device: returns (q int8 [V, H], scale fp32 [V]).  The integers and the
    scales are computed by the library's kernel; torch only provides the two output buffers."""
    if W_lm.dtype != torch.bfloat16 or not W_lm.is_cuda or not W_lm.is_contiguous():
        raise HolaError("hola_quantize_w8 takes a contiguous bfloat16 device tensor")
    lib = load_library()
    V, H = W_lm.shape
    q = torch.empty((V, H), dtype=torch.int8, device=W_lm.device)
    scale = torch.empty((V,), dtype=torch.float32, device=W_lm.device)
    with torch.cuda.device(W_lm.device):
        _check(lib, None, lib.hola_quantize_w8(_dptr(W_lm), V, H, _dptr(q), _dptr(scale), _stream_ptr(stream)),
               "hola_quantize_w8")
    return q, scale


@dataclass
class MixedHead:
    """An LM head stored as groups of 256 vocabulary rows at 4, 8 or 16 bits (HOLA_W_MIXED): the device buffers and the
    hola_wmix struct that points at them.  Keep the object alive while calls that use it are in flight."""
    V: int
    H: int
    widths: list
    W16: torch.Tensor | None
    W8: torch.Tensor | None
    W4: torch.Tensor | None
    shift4: torch.Tensor | None
    w_scale: torch.Tensor
    group_width: torch.Tensor
    group_row: torch.Tensor
    struct: "hola_wmix" = None

    def weight_bytes(self) -> int:
        """Bytes of weights, scales and exponents one pass over the head streams."""
        n = self.w_scale.numel() * 4
        for t in (self.W16, self.W8, self.W4, self.shift4):
            n += 0 if t is None else t.numel() * t.element_size()
        return n


def hola_quantize_mixed(W_lm: torch.Tensor, widths, stream=None) -> MixedHead:
    """bf16 W_lm [V, H] -> the mixed-width form: widths[g] in {4, 8, 16} for group g of 256 vocabulary rows.  Codes,
    scales and exponents are made by one launch of the library's quantiser, to which the widths go as launch parameters (on
    another stream, for widths that are no plain list of integers and beyond 2048 groups: as two tables, in one copy);
    torch provides the buffers."""
    if W_lm.dtype != torch.bfloat16 or not W_lm.is_cuda or not W_lm.is_contiguous():
        raise HolaError("hola_quantize_mixed takes a contiguous bfloat16 device tensor")
    lib = load_library()
    if _host is not None and stream is None:
        st = hola_wmix()
        got = _host.quantize(_entry["hola_quantize_mixed_widths"], W_lm, widths, st, torch._C._cuda_getDevice(), _stream_ptr(None))
        if got is not None:
            _check(lib, None, got[0], "hola_quantize_mixed")
            return MixedHead(*got[1:], st)
    V, H = W_lm.shape
    ng = -(-V // GROUP_ROWS)
    widths = [int(x) for x in widths]
    if len(widths) != ng or not set(widths) <= {4, 8, 16} or H % SUB_BLOCK:
        raise HolaError(f"need {ng} widths out of 4, 8, 16 and H a multiple of {SUB_BLOCK}")
    dev = W_lm.device
    rows = [0] * 17                                              # rows of each width so far
    group_row = array("i")
    for wd in widths:
        group_row.append(rows[wd])
        rows[wd] += GROUP_ROWS
    if ng:
        rows[widths[-1]] -= ng * GROUP_ROWS - V                  # the last group may be ragged
        tables = torch.frombuffer(bytearray(group_row.tobytes() + bytes(widths)), dtype=torch.uint8)
    else:
        tables = torch.empty(0, dtype=torch.uint8)
    s = torch.cuda.current_stream(dev) if stream is None else stream
    if not isinstance(s, torch.cuda.Stream):                     # (as elsewhere, whatever has a cuda_stream)
        s = torch.cuda.ExternalStream(s.cuda_stream, device=dev)
    with torch.cuda.device(dev), torch.cuda.stream(s):
        W16 = torch.empty((rows[16], H), dtype=torch.bfloat16, device=dev) if rows[16] else None
        W8 = torch.empty((rows[8], H), dtype=torch.int8, device=dev) if rows[8] else None
        W4 = torch.empty((rows[4], H // 2), dtype=torch.uint8, device=dev) if rows[4] else None
        shift4 = torch.empty((H // SUB_BLOCK, rows[4]), dtype=torch.uint8, device=dev) if rows[4] else None
        w_scale = torch.empty((V,), dtype=torch.float32, device=dev)
        # (a copy from pageable memory has left that memory when the call returns)
        tables = tables.to(dev, non_blocking=True)
        head = MixedHead(V, H, widths, W16, W8, W4, shift4, w_scale, tables[4 * ng:], tables[:4 * ng].view(torch.int32))
        st = hola_wmix()
        st.W16, st.W8, st.W4, st.shift4 = (t.data_ptr() if t is not None else None for t in (W16, W8, W4, shift4))
        st.group_width, st.group_row = head.group_width.data_ptr(), head.group_row.data_ptr()
        st.rows16, st.rows8, st.rows4 = rows[16], rows[8], rows[4]
        head.struct = st
        if V:
            _check(lib, None, lib.hola_quantize_mixed(_dptr(W_lm), V, H, ctypes.byref(st), _dptr(w_scale), _stream_ptr(s)),
                   "hola_quantize_mixed")
    return head


def hola_lm_head_entropy_static(hidden, W_lm, logits, entropy, logZ, stream=None, status=None) -> None:
    """Steps 1-2 through the entry point that allocates no device memory (no context needed).

    For callers that cannot call cudaMalloc (all of HBM already handed to their own pool, a fixed memory budget,
    an allocator that is locked at this point): the library's only scratch for this call is a 1.25 MiB array
    built into it.  Every tensor is the caller's and lives on the current device: hidden bf16 [B, k+1, H],
    W_lm bf16 [V, H], and the outputs logits fp32 [B, k+1, V], entropy and logZ fp32 [B, k+1].
    At most 512 verify rows (B * (k+1)); larger calls raise HolaError and launch nothing.  Calls share the
    built-in array, so do not let two of them overlap on one GPU.  `status` (int32 [1] on the device, optional) gets
    HOLA_FLAG_TIMEOUT OR-ed in should an on-chip wait run out: it is the only way to learn of that here.
    """
    lib = load_library()
    B, k1, H = hidden.shape
    a = hola_verify_args()
    a.B, a.k, a.H, a.V = B, k1 - 1, H, W_lm.shape[0]
    a.hidden, a.W_lm = _dptr(hidden), _dptr(W_lm)
    a.logits_out, a.entropy, a.logZ = _dptr(logits), _dptr(entropy), _dptr(logZ)
    a.status_word = _dptr(status)
    _check(lib, None, lib.hola_lm_head_entropy_static(ctypes.byref(a), _stream_ptr(stream)),
           "hola_lm_head_entropy_static")


@dataclass
class VerifyOutputs:
    accept_len: torch.Tensor   # int32 [B]
    next_tok: torch.Tensor     # int32 [B]
    entropy: torch.Tensor      # fp32 [B, k+1]
    logZ: torch.Tensor         # fp32 [B, k+1]
    logits: torch.Tensor | None
    status: torch.Tensor       # uint32 as int32 [1]
    draft_entropy: torch.Tensor | None = None   # fp32 [B, k], filled when the gate looks at the draft rows


class _FieldOnDemand:
    """What VerifyOutputs has of a field that an instance lacks: _fresh_outputs leaves out what the call does not fill, and it
    is made when somebody asks.  (Without __set__, so that an instance's own tensor comes first; a __getattr__ would make
    every attribute of every outputs object dearer.)"""

    def __init__(self, name: str):
        self.name = name

    def __get__(self, out, cls=None):
        lazy = None if out is None else out.__dict__.get("_lazy")
        if lazy is None:
            if out is None and self.name == "draft_entropy":
                return None                                      # (the field's default)
            raise AttributeError(f"{cls.__name__!r} object has no attribute {self.name!r}")
        B, k, dev = lazy
        t = (torch.zeros((B, k), dtype=torch.float32, device=dev) if self.name == "draft_entropy"
             else torch.empty(B, dtype=torch.int32, device=dev))
        setattr(out, self.name, t)
        return t


for _name in ("accept_len", "next_tok", "draft_entropy"):
    setattr(VerifyOutputs, _name, _FieldOnDemand(_name))


def _fresh_outputs(ctx: "HolaVerify", B: int, k1: int, want_logits: bool, draws: bool, draft_gate: bool) -> VerifyOutputs:
    """Outputs a call makes for itself: only the tensors that it fills are allocated (one allocation costs the host as
    much as a fifth of a call), the others when somebody asks for them.  The status word is cleared by the call
    (HOLA_ARG_CLEAR_STATUS)."""
    out = VerifyOutputs.__new__(VerifyOutputs)
    dev = ctx._dev
    out._lazy = (B, k1 - 1, dev)
    if _host is not None:
        _host.outputs(out, ctx.device, B, k1, ctx.V, want_logits, draws, draft_gate)
        return out
    # (sizes one by one and empty_like: the cheapest forms, 1.7 and 1.3 us against 2.4 with a tuple)
    out.entropy = e = torch.empty(B, k1, dtype=torch.float32, device=dev)
    out.logZ = torch.empty_like(e)
    out.logits = torch.empty(B, k1, ctx.V, dtype=torch.float32, device=dev) if want_logits else None
    out.status = torch.empty(1, dtype=torch.int32, device=dev)
    if draws:
        out.accept_len = a = torch.empty(B, dtype=torch.int32, device=dev)
        out.next_tok = torch.empty_like(a)
    if draft_gate:
        out.draft_entropy = torch.empty(B, k1 - 1, dtype=torch.float32, device=dev)
    return out


class HolaVerify:
    """Owns one hola_ctx.  Methods are named after the C entry points they call."""

    def __init__(self, maxB: int, maxK: int, H: int, V: int, device: int | None = None):
        if not torch.cuda.is_available():
            raise HolaError("hola_create: no CUDA device; this library has no CPU path")
        self.lib = load_library()
        self.device = torch.cuda.current_device() if device is None else int(device)
        self._dev = torch.device("cuda", self.device)
        self.maxB, self.maxK, self.H, self.V = maxB, maxK, H, V
        self._ctx = ctypes.c_void_p()
        st = self.lib.hola_create(ctypes.byref(self._ctx), self.device, maxB, maxK, H, V)
        _check(self.lib, None, st, "hola_create")

    def close(self):
        if getattr(self, "_ctx", None) and self._ctx.value:
            self.lib.hola_destroy(self._ctx)
            self._ctx = ctypes.c_void_p()

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.close()

    # -------------------------------------------------------------------------------------------------
    def hola_plan(self, B: int, k: int, w_dtype: int = HOLA_W_BF16) -> dict:
        info = hola_plan_info()
        _check(self.lib, self._ctx, self.lib.hola_plan_ex(self._ctx, B, k, w_dtype, ctypes.byref(info)), "hola_plan_ex")
        return {n: getattr(info, n) for n, _ in info._fields_}

    def hola_set_option(self, option: int, value: int):
        _check(self.lib, self._ctx, self.lib.hola_set_option(self._ctx, int(option), int(value)), "hola_set_option")

    def hola_selftest_bounded_wait(self, limit_cycles: int = 100000, stream=None) -> tuple[int, int, int]:
        """Runs the bounded-wait self-test; returns (status word, threads that reached the end, waits that gave up)
        after synchronising the stream."""
        dev = torch.device("cuda", self.device)
        status = torch.zeros(1, dtype=torch.int32, device=dev)
        counters = torch.zeros(2, dtype=torch.int32, device=dev)
        st = self.lib.hola_selftest_bounded_wait(self._ctx, int(limit_cycles), _dptr(status), _dptr(counters),
                                                 _stream_ptr(stream))
        _check(self.lib, self._ctx, st, "hola_selftest_bounded_wait")
        (torch.cuda.current_stream() if stream is None else stream).synchronize()
        return int(status.item()), int(counters[0].item()), int(counters[1].item())

    def hola_selftest_staged_wait(self, limit_cycles: int = 100000, stream=None) -> tuple[int, int, int, int]:
        """Runs the self-test of the wait on staged rows; returns (status word, threads that reached the end, waits that gave
        up, flags that the other CTA reported) after synchronising the stream."""
        status = torch.zeros(1, dtype=torch.int32, device=self._dev)
        counters = torch.zeros(3, dtype=torch.int32, device=self._dev)
        st = self.lib.hola_selftest_staged_wait(self._ctx, int(limit_cycles), _dptr(status), _dptr(counters),
                                                _stream_ptr(stream))
        _check(self.lib, self._ctx, st, "hola_selftest_staged_wait")
        (torch.cuda.current_stream() if stream is None else stream).synchronize()
        return (int(status.item()), *counters.tolist())

    def hola_selftest_mass_wait(self, limit_cycles: int = 100000, stream=None) -> tuple[int, int, int, int, int]:
        """Runs the self-test of the wait on the other CTAs' sums; returns (status word, threads that reached the end, waits
        that gave up, flags that the first CTA reported, CTAs that all sums had reached) after synchronising the stream."""
        status = torch.zeros(1, dtype=torch.int32, device=self._dev)
        counters = torch.zeros(4, dtype=torch.int32, device=self._dev)
        st = self.lib.hola_selftest_mass_wait(self._ctx, int(limit_cycles), _dptr(status), _dptr(counters), _stream_ptr(stream))
        _check(self.lib, self._ctx, st, "hola_selftest_mass_wait")
        (torch.cuda.current_stream() if stream is None else stream).synchronize()
        return (int(status.item()), *counters.tolist())

    def hola_selftest_pace(self, stream=None) -> torch.Tensor:
        """The pace counters of launches that hold several passes, behind what is queued on the stream: zeros between calls."""
        words = torch.empty(HOLA_PACE_WORDS, dtype=torch.int32, device=self._dev)
        _check(self.lib, self._ctx, self.lib.hola_selftest_pace(self._ctx, _dptr(words), _stream_ptr(stream)), "hola_selftest_pace")
        return words

    def hola_selftest_quotient(self, t: torch.Tensor, s: torch.Tensor, stream=None) -> torch.Tensor:
        """t / s (contiguous fp32 tensors on the context's device) as the kernels divide."""
        for x in (t, s):
            if x.dtype != torch.float32 or x.device != self._dev or not x.is_contiguous() or x.numel() != t.numel():
                raise HolaError("hola_selftest_quotient takes two contiguous fp32 tensors of one size on the context's device")
        out = torch.empty_like(t)
        st = self.lib.hola_selftest_quotient(self._ctx, _dptr(t), _dptr(s), t.numel(), _dptr(out), _stream_ptr(stream))
        _check(self.lib, self._ctx, st, "hola_selftest_quotient")
        return out

    def hola_profile_begin(self, max_calls: int):
        _check(self.lib, self._ctx, self.lib.hola_profile_begin(self._ctx, max_calls), "hola_profile_begin")

    def hola_shard_call(self, which: str, args, shard, stream=None):
        """hola_shard_lm_head / hola_shard_accept / hola_shard_sample on prepared argument structs."""
        if which not in ("hola_shard_lm_head", "hola_shard_accept", "hola_shard_sample"):
            raise HolaError(f"unknown entry point {which}")
        st = getattr(self.lib, which)(self._ctx, ctypes.byref(args), ctypes.byref(shard), _stream_ptr(stream))
        _check(self.lib, self._ctx, st, which)

    def hola_host_traffic(self) -> tuple[int, int]:
        """(host-to-device, device-to-host) bytes of the last hola_verify_host call."""
        up, down = ctypes.c_ulonglong(0), ctypes.c_ulonglong(0)
        _check(self.lib, self._ctx, self.lib.hola_host_traffic(self._ctx, ctypes.byref(up), ctypes.byref(down)),
               "hola_host_traffic")
        return int(up.value), int(down.value)

    def hola_profile_end(self, stream=None) -> dict:
        a, b, n = ctypes.c_double(), ctypes.c_double(), ctypes.c_int()
        st = self.lib.hola_profile_end(self._ctx, _stream_ptr(stream), ctypes.byref(a), ctypes.byref(b), ctypes.byref(n))
        _check(self.lib, self._ctx, st, "hola_profile_end")
        return {"lm_head_ms": a.value, "accept_sample_ms": b.value, "calls": n.value}

    def _args(self, hidden, W_lm, draft_tok, draft_q, uniforms, tau, out: VerifyOutputs, B, k,
              gate_source: int = HOLA_GATE_TARGET_ENTROPY, fallback: int = HOLA_FALLBACK_SAMPLE, w_scale=None,
              a8: bool = False, draws: bool = True):
        mixed = W_lm if isinstance(W_lm, MixedHead) else None
        if mixed is not None:
            if mixed.V != self.V or mixed.H != self.H or w_scale is not None or a8:
                raise HolaError("a MixedHead carries its own scales and takes bf16 activations; its shape must be the context's")
            W_lm, w_scale = (mixed.W8 if mixed.W8 is not None else (mixed.W4 if mixed.W4 is not None else mixed.W16)), mixed.w_scale
        if hidden.dtype != torch.bfloat16 or (mixed is None and W_lm.dtype not in (torch.bfloat16, torch.int8)):
            raise HolaError("hidden must be bfloat16, W_lm bfloat16 or int8")
        if mixed is None and (W_lm.dtype == torch.int8) != (w_scale is not None):
            raise HolaError("an int8 W_lm goes with w_scale (fp32 per vocabulary row), a bfloat16 one without")
        if draft_q is not None and draft_q.dtype not in (torch.bfloat16, torch.float32):
            raise HolaError("draft_q must be bfloat16 or float32")
        for t in (hidden, W_lm, draft_tok, draft_q, uniforms):
            if t is not None and not t.is_contiguous():
                raise HolaError("all inputs must be contiguous")
        # (plain integers into the pointer fields: a c_void_p object for each would cost as much as the call itself)
        a = hola_verify_args()
        a.B, a.k, a.H, a.V = B, k, self.H, self.V
        a.hidden = hidden.data_ptr()
        if k > 0:
            if draft_tok is not None:
                a.draft_tok = draft_tok.data_ptr()
            if draft_q is not None:
                a.draft_q = draft_q.data_ptr()
        if draft_q is not None and draft_q.dtype == torch.float32:
            a.q_dtype = HOLA_Q_F32
        if uniforms is not None:
            a.uniforms = uniforms.data_ptr()
        a.tau = float(tau)
        # (an output that is missing stays a null pointer, which the library refuses where it needs it)
        if draws:
            if (t := out.accept_len) is not None:
                a.accept_len = t.data_ptr()
            if (t := out.next_tok) is not None:
                a.next_tok = t.data_ptr()
        if (t := out.entropy) is not None:
            a.entropy = t.data_ptr()
        if (t := out.logZ) is not None:
            a.logZ = t.data_ptr()
        if out.logits is not None:
            a.logits_out = out.logits.data_ptr()
        if out.status is not None:
            a.status_word = out.status.data_ptr()
        a.gate_source, a.fallback = int(gate_source), int(fallback)
        if a.gate_source == HOLA_GATE_DRAFT_ENTROPY and out.draft_entropy is not None:
            a.draft_entropy = out.draft_entropy.data_ptr()
        # a8: True = one 8-bit plane per hidden row (W8A8); "a16" = two planes (16-bit-class activations, W8A16)
        if a8 and w_scale is None:
            raise HolaError("8-bit activation planes (a8) go with an int8 W_lm and its scales")
        if w_scale is not None:
            a.w_scale = w_scale.data_ptr()
        if mixed is not None:
            a.w_dtype, a.wmix = HOLA_W_MIXED, ctypes.addressof(mixed.struct)
        else:
            a.W_lm = W_lm.data_ptr()
            if w_scale is not None:
                a.w_dtype = HOLA_W8A16 if a8 == "a16" else (HOLA_W8A8 if a8 else HOLA_W_INT8)
        return a

    def _native(self, entry, hidden, W_lm, draft_tok, draft_q, uniforms, tau, out, draws, flags, gate_source, fallback, w_scale,
                a8, stream):
        """The call through the native helper: its status, or None where the arguments have to be made from Python."""
        if _host is None or self.lib is not _lib:
            return None
        wmix = 0
        if type(W_lm) is MixedHead:
            if w_scale is not None or a8 or W_lm.V != self.V or W_lm.H != self.H:
                return None
            wmix, w_scale = ctypes.addressof(W_lm.struct), W_lm.w_scale
            W_lm = W_lm.W8 if W_lm.W8 is not None else (W_lm.W4 if W_lm.W4 is not None else W_lm.W16)
        return _host.call(_entry[entry], self._ctx.value, self.H, self.V, hidden, W_lm, draft_tok, draft_q, uniforms, tau, out,
                          draws, flags, gate_source, fallback, w_scale, a8, wmix, _stream_ptr(stream))

    def alloc_outputs(self, B: int, k: int, want_logits: bool = False, device=None) -> VerifyOutputs:
        dev = torch.device("cuda", self.device) if device is None else device
        return VerifyOutputs(
            accept_len=torch.empty(B, dtype=torch.int32, device=dev),
            next_tok=torch.empty(B, dtype=torch.int32, device=dev),
            entropy=torch.empty((B, k + 1), dtype=torch.float32, device=dev),
            logZ=torch.empty((B, k + 1), dtype=torch.float32, device=dev),
            logits=torch.empty((B, k + 1, self.V), dtype=torch.float32, device=dev) if want_logits else None,
            status=torch.zeros(1, dtype=torch.int32, device=dev),
            draft_entropy=torch.zeros((B, k), dtype=torch.float32, device=dev))

    def hola_verify(self, hidden, W_lm, draft_tok, draft_q, uniforms, tau, out: VerifyOutputs | None = None,
                    want_logits: bool = False, stream=None, gate_source: int = HOLA_GATE_TARGET_ENTROPY,
                    fallback: int = HOLA_FALLBACK_SAMPLE, w_scale=None, a8: bool = False) -> VerifyOutputs:
        """The whole verify step on device tensors, asynchronous on the stream.  With w_scale, W_lm is the int8 form
        made by hola_quantize_w8; with a8 as well, the hidden rows are quantised on the fly and the products run on
        the 8-bit tensor-core kind."""
        fresh = not out
        if fresh:
            B, k1 = hidden.shape[:2]
            out = _fresh_outputs(self, B, k1, want_logits, True, gate_source == HOLA_GATE_DRAFT_ENTROPY)
        st = self._native("hola_verify", hidden, W_lm, draft_tok, draft_q, uniforms, tau, out, 1,
                          HOLA_ARG_CLEAR_STATUS if fresh else 0, gate_source, fallback, w_scale, a8, stream)
        if st is None:
            B, k1 = hidden.shape[:2]
            a = self._args(hidden, W_lm, draft_tok, draft_q, uniforms, tau, out, B, k1 - 1, gate_source, fallback, w_scale, a8)
            if fresh:
                a.flags = HOLA_ARG_CLEAR_STATUS
            st = self.lib.hola_verify(self._ctx, ctypes.byref(a), _stream_ptr(stream))
        if st:
            _check(self.lib, self._ctx, st, "hola_verify")
        return out

    def hola_lm_head_entropy(self, hidden, W_lm, out: VerifyOutputs | None = None, want_logits: bool = True,
                             stream=None, w_scale=None, a8: bool = False) -> VerifyOutputs:
        fresh = not out
        if fresh:
            B, k1 = hidden.shape[:2]
            out = _fresh_outputs(self, B, k1, want_logits, False, False)
        st = self._native("hola_lm_head_entropy", hidden, W_lm, None, None, None, 0.0, out, 0,
                          HOLA_ARG_CLEAR_STATUS if fresh else 0, 0, 0, w_scale, a8, stream)
        if st is None:
            B, k1 = hidden.shape[:2]
            a = self._args(hidden, W_lm, None, None, None, 0.0, out, B, k1 - 1, w_scale=w_scale, a8=a8, draws=False)
            if fresh:
                a.flags = HOLA_ARG_CLEAR_STATUS
            st = self.lib.hola_lm_head_entropy(self._ctx, ctypes.byref(a), _stream_ptr(stream))
        if st:
            _check(self.lib, self._ctx, st, "hola_lm_head_entropy")
        return out

    def hola_accept_sample(self, logits, entropy, logZ, draft_tok, draft_q, uniforms, tau, stream=None) -> VerifyOutputs:
        """Steps 3-5 from given fp32 logits [B, k+1, V] and their entropy / logZ."""
        B, k = logits.shape[0], logits.shape[1] - 1
        out = self.alloc_outputs(B, k, False)
        out.logits = logits
        out.entropy.copy_(entropy)
        out.logZ.copy_(logZ)
        a = hola_verify_args()
        a.B, a.k, a.H, a.V = B, k, self.H, self.V
        a.draft_tok = _dptr(draft_tok) if k > 0 else None
        a.draft_q = _dptr(draft_q) if k > 0 else None
        a.q_dtype = HOLA_Q_F32 if (draft_q is not None and draft_q.dtype == torch.float32) else HOLA_Q_BF16
        a.uniforms, a.tau = _dptr(uniforms), float(tau)
        a.accept_len, a.next_tok = _dptr(out.accept_len), _dptr(out.next_tok)
        a.entropy, a.logZ, a.logits_out, a.status_word = _dptr(out.entropy), _dptr(out.logZ), _dptr(logits), _dptr(out.status)
        _check(self.lib, self._ctx, self.lib.hola_accept_sample(self._ctx, ctypes.byref(a), _stream_ptr(stream)),
               "hola_accept_sample")
        return out

    def hola_verify_host(self, hidden, W_lm, draft_tok, draft_q, uniforms, tau, out: VerifyOutputs | None = None,
                         stream=None, gate_source: int = HOLA_GATE_TARGET_ENTROPY,
                         fallback: int = HOLA_FALLBACK_SAMPLE, w_scale=None, a8: bool = False) -> VerifyOutputs:
        """End-to-end form: per-step inputs and all outputs are HOST tensors (pinned for async copies);
        W_lm is the resident device weight.  Returns after the stream has been synchronised."""
        B, k = hidden.shape[0], hidden.shape[1] - 1
        if not isinstance(W_lm, MixedHead) and not W_lm.is_cuda:
            raise HolaError("W_lm must be resident on the device")
        for t in (hidden, draft_tok, draft_q, uniforms):
            if t is not None and not t.is_cpu:
                raise HolaError("hola_verify_host takes host tensors for the per-step inputs")
        out = out or self.alloc_outputs(B, k, False, device=torch.device("cpu"))
        st = None
        if out.logits is None:
            st = self._native("hola_verify_host", hidden, W_lm, draft_tok, draft_q, uniforms, tau, out, 1, 0, gate_source,
                              fallback, w_scale, a8, stream)
        if st is None:
            a = self._args(hidden, W_lm, draft_tok, draft_q, uniforms, tau, out, B, k, gate_source, fallback, w_scale, a8)
            a.logits_out = None
            st = self.lib.hola_verify_host(self._ctx, ctypes.byref(a), _stream_ptr(stream))
        _check(self.lib, self._ctx, st, "hola_verify_host")
        return out


def hola_plan_for_shape(num_sms: int, H: int, V: int, rows: int, w_dtype: int = 0) -> dict:
    """Launch geometry for a shape alone (host arithmetic; needs the library, not a device)."""
    lib = load_library()
    info = hola_plan_info()
    st = lib.hola_plan_for_shape(int(num_sms), int(H), int(V), int(rows), int(w_dtype), ctypes.byref(info))
    if st != 0:
        raise HolaError(f"hola_plan_for_shape: status {st}")
    return {n: getattr(info, n) for n, _ in hola_plan_info._fields_}


def hola_hidden_form_for_shape(num_sms: int, H: int, V: int, rows: int, w_dtype: int = 0) -> int:
    """HOLA_HIDDEN_IN_PLACE, HOLA_HIDDEN_ON_LINES or HOLA_HIDDEN_8BIT: what becomes of the hidden rows ahead of the LM-head
    launch (the last two: by a kernel of its own)."""
    form = ctypes.c_int32()
    st = load_library().hola_hidden_form_for_shape(int(num_sms), int(H), int(V), int(rows), int(w_dtype), ctypes.byref(form))
    if st != 0:
        raise HolaError(f"hola_hidden_form_for_shape: status {st}")
    return form.value


def hola_sample_plan_for_shape(num_sms: int, B: int, k: int, V: int, q_dtype: int = HOLA_Q_BF16,
                               fallback: int = HOLA_FALLBACK_SAMPLE) -> dict:
    """Form of the accept/sample kernel for a shape (host arithmetic; needs the library, not a device)."""
    lib = load_library()
    info = hola_sample_info()
    st = lib.hola_sample_plan_for_shape(int(num_sms), int(B), int(k), int(V), int(q_dtype), int(fallback), ctypes.byref(info))
    if st != 0:
        raise HolaError(f"hola_sample_plan_for_shape: status {st}")
    return {n: getattr(info, n) for n, _ in hola_sample_info._fields_}
