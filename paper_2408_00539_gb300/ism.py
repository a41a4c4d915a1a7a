"""Python binding of libism (ctypes).  Argument marshalling only: every step
of the attention path runs in the library's CUDA kernels.  PyTorch supplies
device memory (outputs and workspaces) and the current CUDA stream.

There is no fallback: if libism.so is missing or a call fails, an exception
is raised.
"""
from __future__ import annotations

import ctypes as C
import functools
import os
import struct
from array import array
from dataclasses import dataclass
from typing import Optional

import numpy as np
import torch

from . import build as _build

ISM_BF16, ISM_FP32, ISM_E4M3 = 0, 1, 2
QUERY, ANSWER = 0, 1
TILE_EMPTY, TILE_FULL, TILE_PARTIAL = 0, 1, 2

_STATUS = {0: "ISM_OK", 1: "ISM_ERR_INVALID_ARG", 2: "ISM_ERR_UNSUPPORTED", 3: "ISM_ERR_CUDA",
           4: "ISM_ERR_TIMEOUT", 5: "ISM_ERR_WORKSPACE"}


class IsmError(RuntimeError):
    def __init__(self, code: int, where: str, detail: str):
        super().__init__(f"{where}: {_STATUS.get(code, code)}: {detail}")
        self.code = code


class _Segments(C.Structure):
    _fields_ = [("num_seqs", C.c_int32), ("num_segs", C.c_int32),
                ("cu_seqlens", C.c_void_p), ("cu_seqlens_host", C.c_void_p),
                ("cu_segs", C.c_void_p), ("cu_segs_host", C.c_void_p),
                ("seg_end", C.c_void_p), ("seg_end_host", C.c_void_p),
                ("seg_type", C.c_void_p), ("seg_type_host", C.c_void_p)]


class _Rope(C.Structure):
    _fields_ = [("cos", C.c_void_p), ("sin", C.c_void_p), ("rows", C.c_int32)]


class _Shape(C.Structure):
    _fields_ = [("num_heads_q", C.c_int32), ("num_heads_kv", C.c_int32), ("head_dim", C.c_int32),
                ("dtype", C.c_int32), ("softmax_scale", C.c_float)]


class _PlanInfo(C.Structure):
    _fields_ = [("fingerprint", C.c_uint64), ("bytes", C.c_size_t)]


EXPORTS = {
    "ism_tile_map_size": (C.c_int, [C.c_void_p, C.c_int32, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p]),
    "ism_build_tile_map": (C.c_int, [C.c_void_p, C.c_int32, C.c_int32] + [C.c_void_p] * 6),
    "ism_attn_fwd_workspace_size": (C.c_int, [C.c_void_p, C.c_void_p, C.c_void_p]),
    "ism_attn_fwd": (C.c_int, [C.c_void_p] * 8 + [C.c_size_t, C.c_void_p]),
    "ism_attn_fwd_e4m3": (C.c_int, [C.c_void_p] * 5 + [C.c_float] * 3 + [C.c_void_p] * 3 + [C.c_size_t, C.c_void_p]),
    "ism_attn_bwd_workspace_size": (C.c_int, [C.c_void_p, C.c_void_p, C.c_void_p]),
    "ism_attn_bwd_workspace_size_min": (C.c_int, [C.c_void_p, C.c_void_p, C.c_void_p]),
    "ism_attn_bwd": (C.c_int, [C.c_void_p] * 12 + [C.c_size_t, C.c_void_p]),
    "ism_attn_fwd_rope": (C.c_int, [C.c_void_p] * 11 + [C.c_size_t, C.c_void_p]),
    "ism_attn_bwd_rope": (C.c_int, [C.c_void_p] * 13 + [C.c_size_t, C.c_void_p]),
    "ism_attn_prefill_append_workspace_size": (C.c_int, [C.c_void_p, C.c_int32, C.c_int32, C.c_void_p]),
    "ism_attn_prefill_append": (C.c_int, [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p, C.c_int32,
                                          C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_int64,
                                          C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p,
                                          C.c_size_t, C.c_void_p]),
    "ism_attn_prefill_append_e4m3": (C.c_int, [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p, C.c_int32,
                                               C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_int64,
                                               C.c_void_p, C.c_void_p, C.c_float, C.c_float, C.c_float, C.c_void_p,
                                               C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p]),
    "ism_attn_prefill_append_paged": (C.c_int, [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p,
                                                C.c_int32, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p,
                                                C.c_int32, C.c_int32, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p,
                                                C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p, C.c_size_t,
                                                C.c_void_p]),
    "ism_attn_prefill_append_rope_workspace_size": (C.c_int, [C.c_void_p, C.c_int32, C.c_int32, C.c_void_p]),
    "ism_attn_prefill_append_rope": (C.c_int, [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p, C.c_int32,
                                               C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_int64,
                                               C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p,
                                               C.c_void_p, C.c_size_t, C.c_void_p]),
    "ism_attn_prefill_append_paged_rope": (C.c_int, [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p,
                                                     C.c_int32, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p,
                                                     C.c_void_p, C.c_int32, C.c_int32, C.c_void_p, C.c_void_p,
                                                     C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p,
                                                     C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p]),
    "ism_attn_prefill_append_e4m3_rope": (C.c_int, [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p,
                                                    C.c_int32, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p,
                                                    C.c_void_p, C.c_int64, C.c_void_p, C.c_void_p, C.c_float,
                                                    C.c_float, C.c_float, C.c_void_p, C.c_void_p, C.c_void_p,
                                                    C.c_void_p, C.c_size_t, C.c_void_p]),
    "ism_check_status": (C.c_int, [C.c_void_p]),
    "ism_debug_timeout_probe": (C.c_int, [C.c_uint32, C.c_void_p]),
    "ism_status_string": (C.c_char_p, [C.c_int]),
    "ism_last_error": (C.c_char_p, []),
    "ism_has_tensor_cores": (C.c_int32, []),
    "ism_set_kernel_timer": (C.c_int, [C.c_int32, C.c_void_p, C.c_void_p]),
    "ism_kernel_launches": (C.c_uint64, []),
    "ism_debug_reload_env": (None, []),
    "ism_debug_mma_tile": (C.c_int, [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p]),
    "ism_debug_mma_tile_e4m3": (C.c_int, [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p]),
    "ism_attn_fwd_noalloc_max_workspace": (C.c_size_t, []),
    "ism_attn_fwd_noalloc": (C.c_int, [C.c_void_p] * 8),
    "ism_attn_plan_size": (C.c_int, [C.c_void_p, C.c_void_p, C.c_void_p]),
    "ism_attn_plan_build": (C.c_int, [C.c_void_p, C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p]),
    "ism_attn_fwd_planned": (C.c_int, [C.c_void_p] * 10),
    "ism_attn_bwd_planned": (C.c_int, [C.c_void_p] * 14 + [C.c_size_t, C.c_void_p]),
    "ism_attn_fwd_rope_planned": (C.c_int, [C.c_void_p] * 13),
    "ism_attn_bwd_rope_planned": (C.c_int, [C.c_void_p] * 15 + [C.c_size_t, C.c_void_p]),
    "ism_call_fwd": (C.c_int, [C.c_char_p]),
    "ism_call_bwd": (C.c_int, [C.c_char_p]),
    "ism_call_pass_sizes": (C.c_int, [C.c_char_p, C.c_int32, C.c_void_p]),
    "ism_call_append": (C.c_int, [C.c_char_p]),
}

# The argument structs of ism_call_* (ism_pass_call_t, ism_append_call_t) as
# packed bytes: one pointer to marshal instead of some twenty arguments.
#   segments; heads, head_dim, dtype, form; scale, descales; rope; plan, fingerprint, bytes;
#   q, k, v, o, lse, dout, dq, dk, dv, q_rot, k_rot; workspace, its bytes; stream
_PASS = struct.Struct("@2i8P5i4d2PiPQN11PPNP")
#   heads, head_dim, dtype, form; scale, descales; rope; batch, l_new, n_new_segs, num_pages, page_size,
#   max_pages; segments; q, k, v, caches; capacity; block tables; cache lengths; o, lse; workspace, its bytes; stream
_APPEND = struct.Struct("@5i4d2Pi4x6i2P5Pq2P2P2PPNP")
_NO_ROPE, _NO_PLAN = (0, 0, 0), (0, 0, 0)
_FORM_E4M3, _FORM_ROPE, _FORM_PAGED = 1, 2, 4

KERNEL_FWD, KERNEL_BWD_DKDV, KERNEL_BWD_DQ, KERNEL_BWD_PRE, KERNEL_DECODE, KERNEL_META, KERNEL_ROPE = 1, 2, 3, 4, 5, 6, 7

_lib = None


def lib_path() -> str:
    return _build.LIB


def load(build_if_missing: bool = False):
    """Load libism.so (building it first when asked)."""
    global _lib
    if _lib is not None:
        return _lib
    path = _build.LIB
    if not os.path.exists(path):
        if not build_if_missing:
            raise RuntimeError(f"libism.so not built ({path}); run __graft_entry__.build()")
        _build.build()
    lib = C.CDLL(path)
    for name, (res, args) in EXPORTS.items():
        fn = getattr(lib, name)
        fn.restype = res
        fn.argtypes = args
    _lib = lib
    return lib


def _check(code: int, where: str):
    if code != 0:
        raise IsmError(code, where, load().ism_last_error().decode())


def _ptr(t: Optional[torch.Tensor]):
    return None if t is None else C.c_void_p(t.data_ptr())


def _stream(device=None):
    return C.c_void_p(torch.cuda.current_stream(device).cuda_stream)


def _raw_stream(t: torch.Tensor) -> int:
    """The current stream of the tensor's device, as an integer."""
    i = t.get_device()
    return torch._C._cuda_getCurrentRawStream(i) if i >= 0 else torch.cuda.current_stream(t.device).cuda_stream


def _addr(a: np.ndarray) -> int:
    return a.__array_interface__["data"][0]


def _host_array(x, dtype, code):
    """(address, length, owner) of a host array of the given element type; the
    owner must outlive the call."""
    if type(x) is list:
        try:
            x = array(code, x)
            return (*x.buffer_info(), x)
        except TypeError:  # other numbers: as numpy converts them
            pass
    x = np.ascontiguousarray(x, dtype=dtype)
    return _addr(x), x.shape[0], x


def _dtype_code(t: torch.Tensor) -> int:
    if t.dtype == torch.bfloat16:
        return ISM_BF16
    if t.dtype == torch.float32:
        return ISM_FP32
    if t.dtype == torch.float8_e4m3fn:
        return ISM_E4M3
    raise TypeError(f"unsupported dtype {t.dtype}")


def _workspace(nbytes: int, device) -> torch.Tensor:
    ws = torch.empty(nbytes, dtype=torch.uint8, device=device)
    if ws.data_ptr() % 256 == 0:  # as the caching allocator hands it out
        return ws
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device=device)
    off = (-ws.data_ptr()) % 256
    return ws[off:off + nbytes]


@dataclass
class Segments:
    """Varlen turn boundaries in both device and host form (the host mirrors
    are used for validation and sizing without a device synchronisation)."""
    cu_seqlens: torch.Tensor
    cu_segs: torch.Tensor
    seg_end: torch.Tensor
    seg_type: torch.Tensor
    cu_seqlens_host: np.ndarray
    cu_segs_host: np.ndarray
    seg_end_host: np.ndarray
    seg_type_host: np.ndarray

    @staticmethod
    def from_numpy(cu_seqlens, cu_segs, seg_end, seg_type, device="cuda") -> "Segments":
        h = [np.ascontiguousarray(cu_seqlens, dtype=np.int32), np.ascontiguousarray(cu_segs, dtype=np.int32),
             np.ascontiguousarray(seg_end, dtype=np.int32), np.ascontiguousarray(seg_type, dtype=np.uint8)]
        d = [torch.from_numpy(x.copy()).to(device) for x in h]
        return Segments(*d, *h)

    @staticmethod
    def from_workload(segs, device="cuda") -> "Segments":
        return Segments.from_numpy(segs.cu_seqlens, segs.cu_segs, segs.seg_end, segs.seg_type, device)

    @property
    def total_tokens(self) -> int:
        return int(self.cu_seqlens_host[-1])

    def fields(self):
        """The values of ism_segments_t, in order."""
        return (self.cu_seqlens_host.shape[0] - 1, self.seg_end_host.shape[0],
                self.cu_seqlens.data_ptr(), _addr(self.cu_seqlens_host), self.cu_segs.data_ptr(),
                _addr(self.cu_segs_host), self.seg_end.data_ptr(), _addr(self.seg_end_host),
                self.seg_type.data_ptr(), _addr(self.seg_type_host))

    def struct(self) -> _Segments:
        s = _Segments()
        s.num_seqs = self.cu_seqlens_host.shape[0] - 1
        s.num_segs = self.seg_end_host.shape[0]
        s.cu_seqlens, s.cu_seqlens_host = self.cu_seqlens.data_ptr(), self.cu_seqlens_host.ctypes.data
        s.cu_segs, s.cu_segs_host = self.cu_segs.data_ptr(), self.cu_segs_host.ctypes.data
        s.seg_end, s.seg_end_host = self.seg_end.data_ptr(), self.seg_end_host.ctypes.data
        s.seg_type, s.seg_type_host = self.seg_type.data_ptr(), self.seg_type_host.ctypes.data
        return s


def _shape(q: torch.Tensor, k: torch.Tensor, scale: float) -> _Shape:
    sh = _Shape()
    sh.num_heads_q, sh.head_dim = q.shape[-2], q.shape[-1]
    sh.num_heads_kv = k.shape[-2]
    sh.dtype = _dtype_code(q)
    sh.softmax_scale = float(scale)
    return sh


def _contig(*ts):
    for t in ts:
        if t is not None and not t.is_contiguous():
            raise ValueError("tensors must be contiguous")


def tile_map(segs: Segments, bm: int = 128, bn: int = 128):
    """Tile map of the segments (device tensors): tile_class, kt_full_end,
    kt_end, qt_begin, kv_end."""
    lib = load()
    s = segs.struct()
    nt, nq, nk = C.c_int64(), C.c_int64(), C.c_int64()
    _check(lib.ism_tile_map_size(C.byref(s), bm, bn, C.byref(nt), C.byref(nq), C.byref(nk)), "ism_tile_map_size")
    dev = segs.cu_seqlens.device
    out = {
        "tile_class": torch.empty(nt.value, dtype=torch.uint8, device=dev),
        "kt_full_end": torch.empty(nq.value, dtype=torch.int32, device=dev),
        "kt_end": torch.empty(nq.value, dtype=torch.int32, device=dev),
        "qt_begin": torch.empty(nk.value, dtype=torch.int32, device=dev),
        "kv_end": torch.empty(segs.total_tokens, dtype=torch.int32, device=dev),
    }
    _check(lib.ism_build_tile_map(C.byref(s), bm, bn, _ptr(out["tile_class"]), _ptr(out["kt_full_end"]),
                                  _ptr(out["kt_end"]), _ptr(out["qt_begin"]), _ptr(out["kv_end"]), _stream(dev)),
           "ism_build_tile_map")
    return out


class Plan:
    """The metadata of one batch of segments (ism_attn_plan_build) for the
    forward and backward of every layer over those segments and head counts:
    built once, passed to fwd / bwd as plan=.  Holds its device buffer, which
    forwards only read; backwards on one plan run one after the other."""

    def __init__(self, segs: Segments, num_heads_q: int, num_heads_kv: int, head_dim: int = 128,
                 dtype: torch.dtype = torch.bfloat16, device="cuda"):
        lib = load()
        self.segs = segs
        probe = torch.empty((0, num_heads_q, head_dim), dtype=dtype)
        self._shape = _shape(probe, torch.empty((0, num_heads_kv, head_dim), dtype=dtype), 1.0)
        n = C.c_size_t()
        _check(lib.ism_attn_plan_size(C.byref(segs.struct()), C.byref(self._shape), C.byref(n)), "ism_attn_plan_size")
        self.buffer = _workspace(n.value, device)
        self.info = _PlanInfo()
        self.build()

    def build(self):
        """Run the metadata pass into the plan (on the current stream)."""
        lib = load()
        _check(lib.ism_attn_plan_build(C.byref(self.segs.struct()), C.byref(self._shape), _ptr(self.buffer),
                                       self.buffer.numel(), C.byref(self.info), _stream(self.buffer.device)),
               "ism_attn_plan_build")
        return self


def _pass_head(segs: Segments, q, k, softmax_scale: float, form: int, descales=(0.0, 0.0, 0.0)):
    """The leading values of ism_pass_call_t."""
    return (*segs.fields(), q.shape[-2], k.shape[-2], q.shape[-1], _dtype_code(q), form, float(softmax_scale),
            *descales)


_NO_TENSORS = (0,) * 14


def _pass_sizes(head, backward: bool):
    """Workspace bytes of the forward, or (full, minimum) of the backward."""
    out = (C.c_size_t * 2)()
    _check(load().ism_call_pass_sizes(_PASS.pack(*head, *_NO_ROPE, *_NO_PLAN, *_NO_TENSORS), backward, out),
           "ism_attn_bwd_workspace_size" if backward else "ism_attn_fwd_workspace_size")
    return (out[0], out[1]) if backward else out[0]


def _plan_fields(plan: "Plan"):
    return (plan.buffer.data_ptr(), plan.info.fingerprint, plan.info.bytes) if plan is not None else _NO_PLAN


def _run_fwd(name, head, rope, plan, q, k, v, out, lse, q_rot, k_rot, workspace):
    """The forward of ism_call_fwd on given outputs; allocates the workspace
    where one is needed and none (or too small a one) is given."""
    ws = (0, 0)
    if plan is None:
        nbytes = _pass_sizes(head, False)
        if workspace is None or workspace.numel() < nbytes:
            workspace = _workspace(nbytes, q.device)
        ws = (workspace.data_ptr(), workspace.numel())
    _check(load().ism_call_fwd(_PASS.pack(
        *head, *rope, *_plan_fields(plan), q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), lse.data_ptr(),
        0, 0, 0, 0, 0 if q_rot is None else q_rot.data_ptr(), 0 if k_rot is None else k_rot.data_ptr(), *ws,
        _raw_stream(q))), name + ("" if plan is None else "_planned"))


def fwd(segs: Segments, q, k, v, softmax_scale: float, out=None, lse=None, workspace=None, plan: Plan = None):
    """Forward over packed dialogues.  q [T,Hq,D], k/v [T,Hkv,D] -> (o, lse [Hq,T]).
    With a plan of these segments the metadata pass is not run again (and no
    workspace is needed)."""
    _contig(q, k, v)
    T, hq, D = q.shape
    if out is None:
        out = torch.empty_like(q)
    if lse is None:
        lse = torch.empty((hq, T), dtype=torch.float32, device=q.device)
    _run_fwd("ism_attn_fwd", _pass_head(segs, q, k, softmax_scale, 0), _NO_ROPE, plan, q, k, v, out, lse, None, None,
             workspace)
    return out, lse


def fwd_e4m3(segs: Segments, q, k, v, q_descale: float, k_descale: float, v_descale: float, softmax_scale: float,
             out=None, lse=None, workspace=None):
    """Forward with e4m3 inputs (torch.float8_e4m3fn; head_dim 128): the
    attention of q * q_descale, k * k_descale, v * v_descale.  Returns
    (o bf16 [T,Hq,D], lse [Hq,T])."""
    _contig(q, k, v)
    T, hq, D = q.shape
    if out is None:
        out = torch.empty(q.shape, dtype=torch.bfloat16, device=q.device)
    if lse is None:
        lse = torch.empty((hq, T), dtype=torch.float32, device=q.device)
    _run_fwd("ism_attn_fwd_e4m3", _pass_head(segs, q, k, softmax_scale, _FORM_E4M3, (q_descale, k_descale, v_descale)),
             _NO_ROPE, None, q, k, v, out, lse, None, None, workspace)
    return out, lse


def fwd_rope(segs: Segments, q, k, v, rope_cos, rope_sin, softmax_scale: float, q_rot=None, k_rot=None, out=None,
             lse=None, workspace=None, plan: "Plan" = None):
    """Forward with rotary encoding: q [T,Hq,D] and k [T,Hkv,D] (unrotated)
    are rotated at their positions inside their sequences (tables rope_cos /
    rope_sin float32 [rows, D/2]) into q_rot / k_rot, then attended.
    Returns (o, lse, q_rot, k_rot); the backward takes q_rot and k_rot."""
    _contig(q, k, v)
    T, hq, D = q.shape
    rope = _rope_fields(rope_cos, rope_sin)
    q_rot = torch.empty_like(q) if q_rot is None else q_rot
    k_rot = torch.empty_like(k) if k_rot is None else k_rot
    out = torch.empty_like(q) if out is None else out
    lse = torch.empty((hq, T), dtype=torch.float32, device=q.device) if lse is None else lse
    _run_fwd("ism_attn_fwd_rope", _pass_head(segs, q, k, softmax_scale, _FORM_ROPE), rope, plan, q, k, v, out, lse,
             q_rot, k_rot, workspace)
    return out, lse, q_rot, k_rot


def _run_bwd(name, head, rope, plan, q, k, v, o, lse, dout, dq, dk, dv, workspace, minimal, fall_back):
    """The backward of ism_call_bwd.  Without a workspace (or with one below
    the minimum) it allocates the full one, or the minimum: with `minimal`, or
    with `fall_back` when the full one does not fit."""
    full, low = _pass_sizes(head, True)
    dq = torch.empty_like(q) if dq is None else dq
    dk = torch.empty_like(k) if dk is None else dk
    dv = torch.empty_like(v) if dv is None else dv
    if workspace is None or workspace.numel() < low:
        try:
            workspace = _workspace(low if minimal else full, q.device)
        except torch.cuda.OutOfMemoryError:
            if minimal or not fall_back:
                raise
            workspace = _workspace(low, q.device)
    _check(load().ism_call_bwd(_PASS.pack(
        *head, *rope, *_plan_fields(plan), q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), lse.data_ptr(),
        dout.data_ptr(), dq.data_ptr(), dk.data_ptr(), dv.data_ptr(), 0, 0, workspace.data_ptr(), workspace.numel(),
        _raw_stream(q))), name + ("" if plan is None else "_planned"))
    return dq, dk, dv


def bwd_rope(segs: Segments, q_rot, k_rot, v, o, lse, dout, rope_cos, rope_sin, softmax_scale: float, dq=None,
             dk=None, dv=None, workspace=None, minimal_workspace: bool = False, plan: "Plan" = None):
    """Backward of ``fwd_rope``: takes the rotated q_rot / k_rot the forward
    wrote and returns (dq, dk, dv) with dq, dk the gradients of the UNROTATED
    queries and keys.  Workspace as for ``bwd``."""
    _contig(q_rot, k_rot, v, o, lse, dout)
    return _run_bwd("ism_attn_bwd_rope", _pass_head(segs, q_rot, k_rot, softmax_scale, _FORM_ROPE),
                    _rope_fields(rope_cos, rope_sin), plan, q_rot, k_rot, v, o, lse, dout, dq, dk, dv, workspace,
                    minimal_workspace, False)


def bwd_workspace_size(segs: Segments, q, k, softmax_scale: float, minimal: bool = False) -> int:
    """Workspace bytes of the backward: the stored-dS schedule's size where
    it applies (else the minimum), or the minimum with minimal=True."""
    lib = load()
    s, sh = segs.struct(), _shape(q, k, softmax_scale)
    nbytes = C.c_size_t()
    fn = "ism_attn_bwd_workspace_size_min" if minimal else "ism_attn_bwd_workspace_size"
    _check(getattr(lib, fn)(C.byref(s), C.byref(sh), C.byref(nbytes)), fn)
    return nbytes.value


def bwd(segs: Segments, q, k, v, o, lse, dout, softmax_scale: float, dq=None, dk=None, dv=None, workspace=None,
        minimal_workspace: bool = False, plan: Plan = None):
    """Backward: (dq, dk, dv) of sum(O * dout).  The library takes the
    stored-dS schedule when the workspace is large enough for it, else the
    recompute schedule.  A given workspace is used as it is (it must hold at
    least the minimum); without one, a workspace of the stored-dS size is
    allocated (the minimum with minimal_workspace=True, or when the larger
    one does not fit in device memory)."""
    _contig(q, k, v, o, lse, dout)
    return _run_bwd("ism_attn_bwd", _pass_head(segs, q, k, softmax_scale, 0), _NO_ROPE, plan, q, k, v, o, lse, dout,
                    dq, dk, dv, workspace, minimal_workspace, True)


@functools.lru_cache(maxsize=256)
def _append_size(hq: int, hkv: int, D: int, dtype: int, batch: int, l_new: int, rope: bool) -> int:
    """Workspace bytes of an append, a function of these numbers alone."""
    sh = _Shape(hq, hkv, D, dtype, 1.0)
    nbytes = C.c_size_t()
    name = "ism_attn_prefill_append_rope_workspace_size" if rope else "ism_attn_prefill_append_workspace_size"
    _check(getattr(load(), name)(C.byref(sh), batch, l_new, C.byref(nbytes)), name)
    return nbytes.value


def append_workspace_size(q_new, k_new, softmax_scale: float, rope: bool = False) -> int:
    """Workspace bytes ``prefill_append`` (``prefill_append_rope`` when rope is
    set) needs for this batch and chunk length."""
    B, Ln, hq, D = q_new.shape
    return _append_size(hq, k_new.shape[-2], D, _dtype_code(q_new), B, Ln, rope)


def _rope_fields(cos, sin):
    """The values of ism_rope_t."""
    _contig(cos, sin)
    if cos.dtype != torch.float32 or sin.dtype != torch.float32 or cos.shape != sin.shape or cos.dim() != 2:
        raise ValueError("rope tables must be float32 [rows, head_dim/2] tensors of one shape")
    return cos.data_ptr(), sin.data_ptr(), cos.shape[0]


def _append(name, form, dtype, q_new, k_new, v_new, k_cache, v_cache, cache_len, cache_len_host, new_seg_end,
            new_seg_type, softmax_scale, out, lse, workspace, rope=_NO_ROPE, descales=(1.0, 1.0, 1.0), capacity=0,
            pages=(0, 0, 0), tables=(0, 0), keep_small=False, prepare=False):
    """One append call (ism_append_call_t); allocates what is not given (a given
    workspace that is too small is replaced unless keep_small).  pages:
    num_pages, page_size, max_pages.  prepare: returns the packed call and what
    its addresses point to instead of running it."""
    B, Ln, hq, D = q_new.shape
    hkv = k_new.shape[-2]
    if out is None:
        out = torch.empty(q_new.shape, dtype=torch.bfloat16 if dtype == ISM_E4M3 else q_new.dtype, device=q_new.device)
    if lse is None:
        lse = torch.empty((hq, B, Ln), dtype=torch.float32, device=q_new.device)
    nbytes = _append_size(hq, hkv, D, dtype, B, Ln, form & _FORM_ROPE)
    if workspace is None or (not keep_small and workspace.numel() < nbytes):
        workspace = _workspace(nbytes, q_new.device)
    end_addr, n_segs, end = _host_array(new_seg_end, np.int32, "i")
    type_addr, _, types = _host_array(new_seg_type, np.uint8, "B")
    len_addr, _, lens = _host_array(cache_len_host, np.int32, "i")
    call = _APPEND.pack(hq, hkv, D, dtype, form, softmax_scale, *descales, *rope, B, Ln, n_segs, *pages, end_addr,
                        type_addr, q_new.data_ptr(), k_new.data_ptr(), v_new.data_ptr(), k_cache.data_ptr(),
                        v_cache.data_ptr(), capacity, *tables, cache_len.data_ptr(), len_addr, out.data_ptr(),
                        lse.data_ptr(), workspace.data_ptr(), workspace.numel(), _raw_stream(q_new))
    if prepare:
        return out, lse, call, (end, types, lens, workspace)
    code = load().ism_call_append(call)
    if code:
        _check(code, name)
    return out, lse


def prefill_append_rope(q_new, k_new, v_new, k_cache, v_cache, cache_len, cache_len_host, new_seg_end, new_seg_type,
                        rope_cos, rope_sin, softmax_scale: float, out=None, lse=None, workspace=None):
    """``prefill_append`` with rotary encoding of the new queries and keys at
    positions cache_len[b] + j (rotate-half pairs, angles given by the fp32
    tables rope_cos / rope_sin [rows, D/2]); the caches receive the rotated
    keys.  Returns (o_new, lse [Hq,B,Ln])."""
    _contig(q_new, k_new, v_new, k_cache, v_cache, cache_len)
    return _append("ism_attn_prefill_append_rope", _FORM_ROPE, _dtype_code(q_new), q_new, k_new, v_new, k_cache, v_cache,
                   cache_len, cache_len_host, new_seg_end, new_seg_type, softmax_scale, out, lse, workspace,
                   _rope_fields(rope_cos, rope_sin), capacity=k_cache.shape[1])


def prefill_append(q_new, k_new, v_new, k_cache, v_cache, cache_len, cache_len_host, new_seg_end, new_seg_type,
                   softmax_scale: float, out=None, lse=None, workspace=None):
    """Append a new turn to the KV caches and attend (Section 2.3).
    q_new [B,Ln,Hq,D], k_new/v_new [B,Ln,Hkv,D], caches [B,cap,Hkv,D],
    cache_len int32 [B] on the device (advanced by Ln), cache_len_host its
    host mirror (the caller advances it).  Returns (o_new, lse [Hq,B,Ln])."""
    _contig(q_new, k_new, v_new, k_cache, v_cache, cache_len)
    return _append("ism_attn_prefill_append", 0, _dtype_code(q_new), q_new, k_new, v_new, k_cache, v_cache, cache_len,
                   cache_len_host, new_seg_end, new_seg_type, softmax_scale, out, lse, workspace,
                   capacity=k_cache.shape[1])


class AppendStep:
    """A prepared ``prefill_append`` call for a generation loop: the arguments
    are marshalled once, so each step is one C call.  The caller keeps the new
    token buffers (q_new, k_new, v_new) and the int32 numpy ``cache_len_host``
    array, refills the buffers before each call and advances the host array in
    place after it (the device ``cache_len`` advances itself)."""

    def __init__(self, q_new, k_new, v_new, k_cache, v_cache, cache_len, cache_len_host: np.ndarray, new_seg_end,
                 new_seg_type, softmax_scale: float, out=None, lse=None, workspace=None, rope=None):
        lib = load()
        _contig(q_new, k_new, v_new, k_cache, v_cache, cache_len)
        if not (isinstance(cache_len_host, np.ndarray) and cache_len_host.dtype == np.int32 and
                cache_len_host.flags["C_CONTIGUOUS"]):
            raise TypeError("cache_len_host must be a contiguous int32 numpy array (advanced in place)")
        self._name = "ism_attn_prefill_append" if rope is None else "ism_attn_prefill_append_rope"
        self.out, self.lse, self._call, kept = _append(
            self._name, 0 if rope is None else _FORM_ROPE, _dtype_code(q_new), q_new, k_new, v_new, k_cache, v_cache,
            cache_len, cache_len_host, new_seg_end, new_seg_type, softmax_scale, out, lse, workspace,
            _NO_ROPE if rope is None else _rope_fields(*rope), capacity=k_cache.shape[1], keep_small=True, prepare=True)
        # what the packed addresses point to
        self._keep = (q_new, k_new, v_new, k_cache, v_cache, cache_len, cache_len_host, rope, kept)
        self._fn = lib.ism_call_append

    def __call__(self):
        code = self._fn(self._call)
        if code:
            _check(code, self._name)
        return self.out, self.lse


def prefill_append_e4m3(q_new, k_new, v_new, k_cache, v_cache, cache_len, cache_len_host, new_seg_end, new_seg_type,
                        q_descale: float, k_descale: float, v_descale: float, softmax_scale: float, out=None, lse=None,
                        workspace=None):
    """``prefill_append`` with e4m3 (torch.float8_e4m3fn) q_new, k_new, v_new and
    caches, dequantised by the per-tensor factors; returns (o bf16, lse)."""
    _contig(q_new, k_new, v_new, k_cache, v_cache, cache_len)
    return _append("ism_attn_prefill_append_e4m3", _FORM_E4M3, _dtype_code(q_new), q_new, k_new, v_new, k_cache, v_cache,
                   cache_len, cache_len_host, new_seg_end, new_seg_type, softmax_scale, out, lse, workspace,
                   keep_small=True, descales=(q_descale, k_descale, v_descale), capacity=k_cache.shape[1])


def _paged(name, form, q_new, k_new, v_new, k_pool, v_pool, page_size, block_table, block_table_host, cache_len,
           cache_len_host, new_seg_end, new_seg_type, softmax_scale, out, lse, workspace, rope=_NO_ROPE):
    _contig(q_new, k_new, v_new, k_pool, v_pool, cache_len, block_table)
    rows = k_pool.shape[0]
    if rows % page_size:
        raise ValueError("pool rows must be a whole number of pages")
    bt = np.ascontiguousarray(block_table_host, dtype=np.int32)
    return _append(name, form | _FORM_PAGED, _dtype_code(q_new), q_new, k_new, v_new, k_pool, v_pool, cache_len,
                   cache_len_host, new_seg_end, new_seg_type, softmax_scale, out, lse, workspace, rope, keep_small=True,
                   pages=(rows // page_size, page_size, block_table.shape[1]),
                   tables=(block_table.data_ptr(), _addr(bt)))


def prefill_append_paged(q_new, k_new, v_new, k_pool, v_pool, page_size: int, block_table, block_table_host,
                         cache_len, cache_len_host, new_seg_end, new_seg_type, softmax_scale: float, out=None,
                         lse=None, workspace=None):
    """``prefill_append`` against a paged cache (Section 2.3): k_pool/v_pool
    [num_pages * page_size, Hkv, D]; key p of sequence b is pool row
    block_table[b, p // page_size] * page_size + p % page_size.  block_table
    int32 [B, max_pages] on the device, block_table_host its host mirror
    (numpy); cache_len / cache_len_host as for ``prefill_append``."""
    return _paged("ism_attn_prefill_append_paged", 0, q_new, k_new, v_new, k_pool, v_pool, page_size, block_table,
                  block_table_host, cache_len, cache_len_host, new_seg_end, new_seg_type, softmax_scale, out, lse,
                  workspace)


def prefill_append_paged_rope(q_new, k_new, v_new, k_pool, v_pool, page_size: int, block_table, block_table_host,
                              cache_len, cache_len_host, new_seg_end, new_seg_type, rope_cos, rope_sin,
                              softmax_scale: float, out=None, lse=None, workspace=None):
    """``prefill_append_paged`` with rotary encoding of the new queries and
    keys at positions cache_len[b] + j (as ``prefill_append_rope``)."""
    return _paged("ism_attn_prefill_append_paged_rope", _FORM_ROPE, q_new, k_new, v_new, k_pool, v_pool, page_size,
                  block_table, block_table_host, cache_len, cache_len_host, new_seg_end, new_seg_type, softmax_scale,
                  out, lse, workspace, _rope_fields(rope_cos, rope_sin))


def prefill_append_e4m3_rope(q_new, k_new, v_new, k_cache, v_cache, cache_len, cache_len_host, new_seg_end,
                             new_seg_type, q_descale: float, k_descale: float, v_descale: float, rope_cos, rope_sin,
                             softmax_scale: float, out=None, lse=None, workspace=None):
    """Rotary append against e4m3 caches: q_new, k_new, v_new are bf16 and
    unrotated; queries and keys are rotated at positions cache_len[b] + j,
    then quantised with the factors (keys and values into the caches).
    Returns (o bf16, lse [Hq,B,Ln])."""
    _contig(q_new, k_new, v_new, k_cache, v_cache, cache_len)
    return _append("ism_attn_prefill_append_e4m3_rope", _FORM_E4M3 | _FORM_ROPE, ISM_E4M3, q_new, k_new, v_new, k_cache,
                   v_cache, cache_len, cache_len_host, new_seg_end, new_seg_type, softmax_scale, out, lse, workspace,
                   _rope_fields(rope_cos, rope_sin), keep_small=True, descales=(q_descale, k_descale, v_descale),
                   capacity=k_cache.shape[1])


def debug_mma_tile_e4m3(a: torch.Tensor, b: torch.Tensor, mode: int) -> torch.Tensor:
    """One 128x128x128 e4m3 tcgen05 tile product (diagnostic): mode 0 a @ b.T,
    mode 1 a @ b, mode 2 a @ b with a in tensor memory; a, b float8_e4m3fn."""
    c = torch.empty((128, 128), dtype=torch.float32, device=a.device)
    _check(load().ism_debug_mma_tile_e4m3(_ptr(a), _ptr(b), _ptr(c), mode, _stream(a.device)),
           "ism_debug_mma_tile_e4m3")
    return c


def check_status(device=None):
    """Synchronise the current stream and raise if a kernel gave up a wait."""
    _check(load().ism_check_status(_stream(device)), "ism_check_status")


def debug_timeout_probe(spin_limit: int = 64, device=None) -> int:
    """Run the bounded-wait probe; returns the status code ism_check_status
    reports afterwards (expected ISM_ERR_TIMEOUT = 4)."""
    lib = load()
    _check(lib.ism_debug_timeout_probe(spin_limit, _stream(device)), "ism_debug_timeout_probe")
    return lib.ism_check_status(_stream(device))


def has_tensor_cores() -> bool:
    return bool(load().ism_has_tensor_cores())


def set_kernel_timer(kernel_id: int, start: "torch.cuda.Event" = None, stop: "torch.cuda.Event" = None):
    """Bracket every launch of one kernel kind (on this thread) with the
    given CUDA events; call with no events to clear."""
    sp = None if start is None else C.c_void_p(start.cuda_event)
    ep = None if stop is None else C.c_void_p(stop.cuda_event)
    _check(load().ism_set_kernel_timer(kernel_id, sp, ep), "ism_set_kernel_timer")


def kernel_launches() -> int:
    return int(load().ism_kernel_launches())


def debug_mma_tile(a: torch.Tensor, b: torch.Tensor, mode: int) -> torch.Tensor:
    """One 128x128x128 tcgen05 tile product (diagnostic): mode 0/2/4 a @ b.T,
    mode 1/3/5 a @ b, mode 6/7 a.T @ b; modes 2/3 stage operands with TMA,
    4/5 put a in tensor memory, 7 stages a 8-interleaved; mode + 8 issues the
    k-steps through the batched one-election form."""
    c = torch.empty((128, 128), dtype=torch.float32, device=a.device)
    _check(load().ism_debug_mma_tile(_ptr(a), _ptr(b), _ptr(c), mode, _stream(a.device)), "ism_debug_mma_tile")
    return c
