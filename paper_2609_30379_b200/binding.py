"""ctypes binding of libnested_pair.so: argument marshalling only.

Every function here has the name of the C entry point it calls (include/nested_pair.h) and does
nothing but convert torch tensors to device pointers and check the returned status.  torch is
used for device memory and streams; all arithmetic runs in the library's CUDA kernels.  If the
shared library is missing the import fails: there is no CPU or eager fallback.
"""
from __future__ import annotations

import ctypes as C
import os
from typing import Optional, Sequence

import numpy as np
import torch

from . import build as _build

NT_OK = 0
NT_F32, NT_BF16 = 0, 1
NT_ORDER_TOKEN_NC, NT_ORDER_PAIR_IJC = 0, 1
NT_REDUCE_MEAN, NT_REDUCE_SUM = 0, 1
NT_OP_PAIR_BROADCAST, NT_OP_TRI_MUL_OUT, NT_OP_ROW_ATTN, NT_OP_BLOCK = 0, 1, 2, 3

STATUS_NAMES = {0: "NT_OK", 1: "NT_ERR_INVALID_ARG", 2: "NT_ERR_UNSUPPORTED", 3: "NT_ERR_WORKSPACE",
                4: "NT_ERR_CUDA", 5: "NT_ERR_TIMEOUT", 6: "NT_ERR_INCONSISTENT"}

EXPORTS = ("nt_offsets_build", "nt_pair_broadcast", "nt_pair_broadcast_add", "nt_pair_broadcast_static", "nt_tri_mul_out", "nt_tri_mul_in",
           "nt_row_attn_pairbias", "nt_row_attn_pairbias_mean", "nt_col_attn_pairbias", "nt_single_attn_pairbias",
           "nt_single_attn_workspace_bytes", "nt_rect_offsets_build", "nt_rect_pair_broadcast",
           "nt_rect_broadcast_workspace_bytes", "nt_segment_reduce", "nt_pair_transition", "nt_transition_workspace_bytes", "nt_token_update",
           "nt_workspace_bytes", "nt_status_string",
           "nt_prepare_trimul_weights", "nt_prepare_attn_weights", "nt_launch_count", "nt_force_generic", "nt_debug_bounds_report", "nt_attn_core_mode", "nt_debug_attn_drop", "nt_debug_expire_wait", "nt_bench_exp_rate", "nt_profile_begin", "nt_profile_end")


class NtError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {STATUS_NAMES.get(status, status)}")


class nt_layout(C.Structure):
    _fields_ = [("B", C.c_int32), ("T1", C.c_int64), ("T2", C.c_int64),
                ("lengths_h", C.c_void_p), ("lengths_d", C.c_void_p), ("tok_off_d", C.c_void_p),
                ("pair_off_d", C.c_void_p), ("row_splits_d", C.c_void_p), ("status_d", C.c_void_p)]


class nt_trimul_weights(C.Structure):
    _fields_ = [(n, C.c_void_p) for n in ("ln_in_gamma", "ln_in_beta", "W_ap", "W_ag", "W_bp", "W_bg", "W_g",
                                          "ln_out_gamma", "ln_out_beta", "W_o", "prepared")]


class nt_attn_weights(C.Structure):
    _fields_ = [(n, C.c_void_p) for n in ("ln_gamma", "ln_beta", "W_q", "W_k", "W_v", "W_b", "W_g", "W_o", "prepared")]


class nt_single_attn_weights(C.Structure):
    _fields_ = [(n, C.c_void_p) for n in ("ln_gamma", "ln_beta", "W_q", "W_k", "W_v", "W_g", "W_o", "ln_z_gamma",
                                          "ln_z_beta", "W_b")]


class nt_transition_weights(C.Structure):
    _fields_ = [(k, C.c_void_p) for k in ("ln_gamma", "ln_beta", "W_a", "W_b", "W_2")]


# the names of a weights structure's fields, in order
_TRIMUL, _ATTN, _SINGLE = (tuple(n for n, _ in t._fields_) for t in (nt_trimul_weights, nt_attn_weights, nt_single_attn_weights))


def _load() -> C.CDLL:
    # NESTED_PAIR_LIB selects another build of the library (the checked one, for instance)
    path = os.environ.get("NESTED_PAIR_LIB") or _build.LIB_PATH
    if not os.path.exists(path):
        raise ImportError(f"{path} is missing: build it with __graft_entry__.build() "
                          "(python -m paper_2609_30379_b200.build); there is no fallback path")
    lib = C.CDLL(path)
    vp, i32, i64, f32, sz = C.c_void_p, C.c_int32, C.c_int64, C.c_float, C.c_size_t
    lib.nt_offsets_build.argtypes = [vp, i32, i64, i64, vp, vp, vp, vp, vp, vp, vp, vp, vp, vp]
    lib.nt_pair_broadcast.argtypes = [C.POINTER(nt_layout), i32, i32, i32, vp, vp, vp, vp, vp, f32, vp, vp, sz, vp]
    lib.nt_pair_broadcast_add.argtypes = lib.nt_pair_broadcast.argtypes
    lib.nt_pair_broadcast_static.argtypes = [C.POINTER(nt_layout), i32, i32, i32, vp, vp, vp, vp, vp, f32, vp, vp]
    lib.nt_tri_mul_out.argtypes = [C.POINTER(nt_layout), i32, i32, i32, C.POINTER(nt_trimul_weights), f32, vp, vp, sz, vp]
    lib.nt_tri_mul_in.argtypes = lib.nt_tri_mul_out.argtypes
    lib.nt_single_attn_pairbias.argtypes = [C.POINTER(nt_layout), i32, i32, i32, i32, i32, C.POINTER(nt_single_attn_weights),
                                            f32, vp, vp, vp, sz, vp]
    lib.nt_single_attn_workspace_bytes.argtypes = [i32, vp, i32, i32, i32, i32]
    lib.nt_single_attn_workspace_bytes.restype = sz
    lib.nt_rect_offsets_build.argtypes = [vp, vp, i32, i64, i64, i64, vp, vp, vp, vp, vp, vp, vp, vp, vp]
    lib.nt_rect_offsets_build.restype = i32
    lib.nt_rect_pair_broadcast.argtypes = [i32, i32, vp, vp, i32, i32, vp, vp, vp, vp, vp, vp, f32, vp, vp, sz, vp]
    lib.nt_rect_pair_broadcast.restype = i32
    lib.nt_rect_broadcast_workspace_bytes.argtypes = [vp, vp, i32, i32]
    lib.nt_rect_broadcast_workspace_bytes.restype = sz
    lib.nt_col_attn_pairbias.argtypes = [C.POINTER(nt_layout), i32, i32, i32, i32, C.POINTER(nt_attn_weights), f32, vp, vp, sz, vp]
    lib.nt_row_attn_pairbias_mean.argtypes = [C.POINTER(nt_layout), i32, i32, i32, i32, C.POINTER(nt_attn_weights), f32, vp, vp, vp, sz, vp]
    lib.nt_row_attn_pairbias.argtypes = [C.POINTER(nt_layout), i32, i32, i32, i32, i32, C.POINTER(nt_attn_weights),
                                         f32, vp, vp, sz, vp]
    lib.nt_segment_reduce.argtypes = [i32, i32, i32, i64, i64, vp, vp, vp, vp, vp]
    lib.nt_token_update.argtypes = [i32, i32, i32, i64, vp, vp, vp, vp]
    lib.nt_pair_transition.argtypes = [i32, i32, i32, i64, C.POINTER(nt_transition_weights), f32, vp, vp, sz, vp, vp]
    lib.nt_pair_transition.restype = i32
    lib.nt_transition_workspace_bytes.argtypes = [i32, i32, i32, i64]
    lib.nt_transition_workspace_bytes.restype = sz
    lib.nt_workspace_bytes.argtypes = [i32, i32, i32, vp, i32, vp]
    lib.nt_workspace_bytes.restype = sz
    lib.nt_status_string.argtypes = [i32]
    lib.nt_status_string.restype = C.c_char_p
    lib.nt_launch_count.argtypes = []
    lib.nt_launch_count.restype = i64
    lib.nt_prepare_trimul_weights.argtypes = [i32, i32, i32, vp, vp, sz, vp]
    lib.nt_prepare_trimul_weights.restype = i32
    lib.nt_prepare_attn_weights.argtypes = [i32, i32, i32, i32, vp, vp, sz, vp]
    lib.nt_prepare_attn_weights.restype = i32
    lib.nt_force_generic.argtypes = [i32]
    lib.nt_force_generic.restype = i32
    lib.nt_debug_expire_wait.argtypes = [vp, C.c_int64, vp, vp]
    lib.nt_debug_expire_wait.restype = i32
    lib.nt_bench_exp_rate.argtypes = [i32, i32, i32, vp, vp, vp]
    lib.nt_bench_exp_rate.restype = i32
    lib.nt_debug_bounds_report.argtypes = [vp, i32]
    lib.nt_debug_bounds_report.restype = i32
    lib.nt_attn_core_mode.argtypes = [i32]
    lib.nt_attn_core_mode.restype = i32
    lib.nt_debug_attn_drop.argtypes = [i32]
    lib.nt_debug_attn_drop.restype = i32
    lib.nt_profile_begin.argtypes = []
    lib.nt_profile_begin.restype = i32
    lib.nt_profile_end.argtypes = [vp, sz, vp, vp, i32]
    lib.nt_profile_end.restype = i32
    for name in ("nt_offsets_build", "nt_pair_broadcast", "nt_pair_broadcast_add", "nt_pair_broadcast_static", "nt_tri_mul_out", "nt_tri_mul_in",
                 "nt_row_attn_pairbias", "nt_row_attn_pairbias_mean", "nt_col_attn_pairbias", "nt_single_attn_pairbias",
                 "nt_segment_reduce", "nt_token_update"):
        getattr(lib, name).restype = i32
    return lib


lib = _load()


def _ptr(t: Optional[torch.Tensor]):
    if t is None:
        return None
    if not t.is_cuda:
        raise ValueError("device tensor expected")
    if not t.is_contiguous():
        raise ValueError("contiguous tensor expected")
    return t.data_ptr()


# the current stream's handle without building a Stream object (0.2 us instead of 3, several times a pass)
_current_device, _current_raw_stream = torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream


def _stream(stream):
    return _current_raw_stream(_current_device()) if stream is None else stream.cuda_stream


def _check(st: int, where: str):
    if st != NT_OK:
        raise NtError(st, where)


def dtype_code(t: torch.dtype) -> int:
    if t == torch.float32:
        return NT_F32
    if t == torch.bfloat16:
        return NT_BF16
    raise ValueError(f"unsupported dtype {t}")


class Layout:
    """Host lengths plus the device mirrors of one batch; owns the buffers nt_layout points at."""

    def __init__(self, lengths: Sequence[int], device="cuda", stream=None, with_maps: bool = False):
        self.lengths_h = np.ascontiguousarray(np.asarray(lengths, dtype=np.int64))
        self.B = int(self.lengths_h.shape[0])
        self.T1 = int(self.lengths_h.sum())
        self.T2 = int(np.dot(self.lengths_h, self.lengths_h))
        dev = torch.device(device)
        if torch.cuda.is_current_stream_capturing():
            raise RuntimeError("a Layout uploads its lengths: build it before the capture begins")
        # one allocation for all offset arrays, each on a multiple of 16 bytes; the zeroed status word and the lengths in
        # front of it arrive in one copy
        odd = self.B & 1
        sizes = (1, 1, self.B, odd, self.B + 1, 1 - odd, self.B + 1, 1 - odd, self.T1 + 1)
        buf = torch.empty(sum(sizes), dtype=torch.int64, device=dev)
        status, _, self.lengths_d, _, self.tok_off, _, self.pair_off, _, self.row_splits = buf.split(sizes)
        self.status = status.view(torch.int32)[:1]
        head = np.zeros(2 + self.B, dtype=np.int64)
        head[2:] = self.lengths_h
        # On the caller's own stream the copy is enqueued like the kernels that read it (a blocking copy would drain the
        # stream for every new batch).  Kernels on another stream must not start before the current one is through with
        # whatever had this memory, so there the copy blocks.
        buf[:2 + self.B].copy_(torch.from_numpy(head), non_blocking=stream is None)
        self.pos_sample = self.pos_i = self.pos_j = self.gather_rows = self.gather_cols = None
        if with_maps:
            self.pos_sample = torch.empty(self.T2, dtype=torch.int32, device=dev)
            self.pos_i = torch.empty(self.T2, dtype=torch.int32, device=dev)
            self.pos_j = torch.empty(self.T2, dtype=torch.int32, device=dev)
            self.gather_rows = torch.empty(self.T2, dtype=torch.int64, device=dev)
            self.gather_cols = torch.empty(self.T2, dtype=torch.int64, device=dev)
        nt_offsets_build(self.lengths_d, self.B, self.T1, self.T2, self.tok_off, self.pair_off, self.row_splits,
                         self.pos_sample, self.pos_i, self.pos_j, self.gather_rows, self.gather_cols,
                         self.status, stream)
        if stream is not None:      # dropping the Layout must not hand its memory out before that stream is done with it
            user = stream if isinstance(stream, torch.cuda.Stream) else torch.cuda.ExternalStream(stream.cuda_stream, device=dev)
            for t in (buf, self.pos_sample, self.pos_i, self.pos_j, self.gather_rows, self.gather_cols):
                if t is not None:
                    t.record_stream(user)
        self.c = nt_layout(self.B, self.T1, self.T2, self.lengths_h.ctypes.data if self.B else None,
                           _ptr(self.lengths_d) if self.B else None, _ptr(self.tok_off), _ptr(self.pair_off),
                           _ptr(self.row_splits), _ptr(self.status))

    def rebuild(self, lengths: Sequence[int], stream=None):
        """Takes the lengths of another batch with the same B, T1 and T2 (the buffer sizes) and builds its offsets
        into the same device buffers, so that pointers held elsewhere (a captured graph, a cached nt_layout) stay valid."""
        new = np.ascontiguousarray(np.asarray(lengths, dtype=np.int64))
        if new.shape != self.lengths_h.shape or int(new.sum()) != self.T1 or int((new * new).sum()) != self.T2:
            raise ValueError("Layout.rebuild needs the same B, T1 and T2; build a new Layout instead")
        np.copyto(self.lengths_h, new)
        if self.B:      # (blocking for kernels on another stream, as above)
            self.lengths_d.copy_(torch.from_numpy(self.lengths_h), non_blocking=stream is None)
        nt_offsets_build(self.lengths_d, self.B, self.T1, self.T2, self.tok_off, self.pair_off, self.row_splits,
                         self.pos_sample, self.pos_i, self.pos_j, self.gather_rows, self.gather_cols,
                         self.status, stream)

    def device_status(self) -> int:
        return int(self.status.item())


def nt_offsets_build(lengths_d, B, T1, T2, tok_off_d, pair_off_d, row_splits_d=None, pos_sample_d=None,
                     pos_i_d=None, pos_j_d=None, gather_rows_d=None, gather_cols_d=None, status_d=None, stream=None):
    st = lib.nt_offsets_build(_ptr(lengths_d) if B else None, B, T1, T2, _ptr(tok_off_d), _ptr(pair_off_d),
                              _ptr(row_splits_d), _ptr(pos_sample_d), _ptr(pos_i_d), _ptr(pos_j_d),
                              _ptr(gather_rows_d), _ptr(gather_cols_d), _ptr(status_d), _stream(stream))
    _check(st, "nt_offsets_build")


def nt_workspace_bytes(op: int, dt: int, order: int, lengths_h: np.ndarray, dims: Sequence[int]) -> int:
    lengths_h = np.ascontiguousarray(lengths_h, dtype=np.int64)
    d = (C.c_int32 * 5)(*[int(v) for v in dims])
    return int(lib.nt_workspace_bytes(op, dt, order, lengths_h.ctypes.data, int(lengths_h.shape[0]), C.addressof(d)))


def nt_pair_broadcast(L: Layout, x, W_a, W_b, ln_gamma, ln_beta, ln_eps, z, workspace, stream=None):
    c_s, c_z = int(W_a.shape[1]), int(W_a.shape[0])
    st = lib.nt_pair_broadcast(C.byref(L.c), dtype_code(x.dtype), c_s, c_z, _ptr(x), _ptr(W_a), _ptr(W_b),
                               _ptr(ln_gamma), _ptr(ln_beta), float(ln_eps), _ptr(z), _ptr(workspace),
                               workspace.nbytes, _stream(stream))
    _check(st, "nt_pair_broadcast")


def nt_pair_broadcast_add(L: Layout, x, W_a, W_b, ln_gamma, ln_beta, ln_eps, z, workspace, stream=None):
    c_s, c_z = int(W_a.shape[1]), int(W_a.shape[0])
    st = lib.nt_pair_broadcast_add(C.byref(L.c), dtype_code(x.dtype), c_s, c_z, _ptr(x), _ptr(W_a), _ptr(W_b),
                               _ptr(ln_gamma), _ptr(ln_beta), float(ln_eps), _ptr(z), _ptr(workspace),
                               workspace.nbytes, _stream(stream))
    _check(st, "nt_pair_broadcast_add")


def nt_pair_broadcast_static(L: Layout, x, W_a, W_b, ln_gamma, ln_beta, ln_eps, z, stream=None):
    """nt_pair_broadcast with the scratch in the library's own fixed device array: for callers that
    cannot allocate a workspace.  Raises NtError(NT_ERR_WORKSPACE) when the batch exceeds that array."""
    c_s, c_z = int(W_a.shape[1]), int(W_a.shape[0])
    st = lib.nt_pair_broadcast_static(C.byref(L.c), dtype_code(x.dtype), c_s, c_z, _ptr(x), _ptr(W_a), _ptr(W_b),
                                      _ptr(ln_gamma), _ptr(ln_beta), float(ln_eps), _ptr(z), _stream(stream))
    _check(st, "nt_pair_broadcast_static")


def nt_tri_mul_out(L: Layout, W: dict, ln_eps, z, workspace, stream=None):
    c_h, c_z = int(W["W_ap"].shape[0]), int(W["W_ap"].shape[1])
    w = nt_trimul_weights(*[_ptr(W[n]) if n != "prepared" else _ptr(W.get(n)) for n in _TRIMUL])
    st = lib.nt_tri_mul_out(C.byref(L.c), dtype_code(z.dtype), c_z, c_h, C.byref(w), float(ln_eps), _ptr(z),
                            _ptr(workspace), workspace.nbytes, _stream(stream))
    _check(st, "nt_tri_mul_out")


def nt_tri_mul_in(L: Layout, W: dict, ln_eps, z, workspace, stream=None):
    """Incoming direction of the triangle update; same arguments and workspace as nt_tri_mul_out."""
    c_h, c_z = int(W["W_ap"].shape[0]), int(W["W_ap"].shape[1])
    w = nt_trimul_weights(*[_ptr(W[n]) if n != "prepared" else _ptr(W.get(n)) for n in _TRIMUL])
    st = lib.nt_tri_mul_in(C.byref(L.c), dtype_code(z.dtype), c_z, c_h, C.byref(w), float(ln_eps), _ptr(z),
                           _ptr(workspace), workspace.nbytes, _stream(stream))
    _check(st, "nt_tri_mul_in")


def nt_row_attn_pairbias(L: Layout, order: int, W: dict, H: int, d: int, ln_eps, zx, workspace, stream=None):
    c = int(W["W_q"].shape[1])
    w = nt_attn_weights(*[_ptr(W.get(n)) for n in _ATTN])
    st = lib.nt_row_attn_pairbias(C.byref(L.c), order, dtype_code(zx.dtype), c, H, d, C.byref(w), float(ln_eps),
                                  _ptr(zx), _ptr(workspace), workspace.nbytes,
                                  _stream(stream))
    _check(st, "nt_row_attn_pairbias")


def nt_single_attn_pairbias(L: Layout, W: dict, H: int, d: int, ln_eps, x, z, workspace, stream=None):
    """Pair-biased single attention: x [T1, c_s] updated in place, z [T2, c_z] read only."""
    c_s, c_z = int(W["W_q"].shape[1]), int(W["W_b"].shape[1])
    w = nt_single_attn_weights(*[_ptr(W[n]) for n in _SINGLE])
    st = lib.nt_single_attn_pairbias(C.byref(L.c), dtype_code(x.dtype), c_s, c_z, H, d, C.byref(w), float(ln_eps),
                                     _ptr(x), _ptr(z), _ptr(workspace), workspace.nbytes,
                                     _stream(stream))
    _check(st, "nt_single_attn_pairbias")


def nt_single_attn_workspace_bytes(dtype, lengths, c_s: int, H: int, d: int) -> int:
    arr = (C.c_int64 * max(len(lengths), 1))(*[int(v) for v in lengths])
    return int(lib.nt_single_attn_workspace_bytes(dtype_code(dtype), arr, len(lengths), c_s, H, d))


class RectLayout:
    """Device offsets of a batch of rectangular pairs (N_s, M_s): tokn_off, tokm_off, pair_off, the level-2 row
    splits and (optionally) the cell decode, all built on the device by nt_rect_offsets_build."""

    def __init__(self, lengths_n, lengths_m, with_maps=False, device="cuda", stream=None):
        import torch
        self.lengths_n = [int(v) for v in lengths_n]
        self.lengths_m = [int(v) for v in lengths_m]
        assert len(self.lengths_n) == len(self.lengths_m)
        self.B = len(self.lengths_n)
        self.T1n, self.T1m = sum(self.lengths_n), sum(self.lengths_m)
        self.T2 = sum(n * m for n, m in zip(self.lengths_n, self.lengths_m))
        self.ln_h = (C.c_int64 * max(self.B, 1))(*self.lengths_n)
        self.lm_h = (C.c_int64 * max(self.B, 1))(*self.lengths_m)
        i64t = dict(dtype=torch.int64, device=device)
        self.ln_d = torch.tensor(self.lengths_n, **i64t)
        self.lm_d = torch.tensor(self.lengths_m, **i64t)
        self.tokn_off = torch.empty(self.B + 1, **i64t)
        self.tokm_off = torch.empty(self.B + 1, **i64t)
        self.pair_off = torch.empty(self.B + 1, **i64t)
        self.row_splits = torch.empty(self.T1n + 1, **i64t)
        self.status = torch.zeros(1, dtype=torch.int32, device=device)
        self.pos_sample = self.pos_i = self.pos_j = None
        if with_maps:
            self.pos_sample = torch.empty(self.T2, dtype=torch.int32, device=device)
            self.pos_i = torch.empty(self.T2, dtype=torch.int32, device=device)
            self.pos_j = torch.empty(self.T2, dtype=torch.int32, device=device)
        st = lib.nt_rect_offsets_build(_ptr(self.ln_d) if self.B else None, _ptr(self.lm_d) if self.B else None, self.B, self.T1n,
                                       self.T1m, self.T2, _ptr(self.tokn_off), _ptr(self.tokm_off), _ptr(self.pair_off),
                                       _ptr(self.row_splits), _ptr(self.pos_sample), _ptr(self.pos_i), _ptr(self.pos_j),
                                       _ptr(self.status), _stream(stream))
        _check(st, "nt_rect_offsets_build")

    def device_status(self) -> int:
        return int(self.status.item())


def nt_rect_broadcast_workspace_bytes(L: RectLayout, c_z: int) -> int:
    return int(lib.nt_rect_broadcast_workspace_bytes(L.ln_h, L.lm_h, L.B, c_z))


def nt_rect_pair_broadcast(L: RectLayout, x, y, W_a, W_b, ln_gamma, ln_beta, ln_eps, z, workspace, stream=None):
    """Rectangular broadcast from row tokens x [T1n, c_s] and column tokens y [T1m, c_s] into z [T2, c_z]."""
    c_s, c_z = int(W_a.shape[1]), int(W_a.shape[0])
    st = lib.nt_rect_pair_broadcast(dtype_code(x.dtype), L.B, L.ln_h, L.lm_h, c_s, c_z, _ptr(x), _ptr(y), _ptr(W_a), _ptr(W_b),
                                    _ptr(ln_gamma), _ptr(ln_beta), float(ln_eps), _ptr(z), _ptr(workspace),
                                    workspace.nbytes, _stream(stream))
    _check(st, "nt_rect_pair_broadcast")


def nt_row_attn_pairbias_mean(L: Layout, W: dict, H: int, d: int, ln_eps, z, m_out, workspace, stream=None):
    """Row-wise pair-biased attention in pair order followed by the mean over j of the updated state into
    m_out [T1, c], in one call (the column sums come from the output stage's tiles where that stage runs)."""
    c = int(W["W_q"].shape[1])
    w = nt_attn_weights(*[_ptr(W.get(n)) for n in _ATTN])
    st = lib.nt_row_attn_pairbias_mean(C.byref(L.c), dtype_code(z.dtype), c, H, d, C.byref(w), float(ln_eps),
                                       _ptr(z), _ptr(m_out), _ptr(workspace),
                                       workspace.nbytes, _stream(stream))
    _check(st, "nt_row_attn_pairbias_mean")


def nt_col_attn_pairbias(L: Layout, W: dict, H: int, d: int, ln_eps, z, workspace, stream=None):
    """Column-wise ("ending node") pair-biased attention on the packed pair state; weights and workspace as for
    nt_row_attn_pairbias in pair order."""
    c = int(W["W_q"].shape[1])
    w = nt_attn_weights(*[_ptr(W.get(n)) for n in _ATTN])
    st = lib.nt_col_attn_pairbias(C.byref(L.c), dtype_code(z.dtype), c, H, d, C.byref(w), float(ln_eps),
                                  _ptr(z), _ptr(workspace), workspace.nbytes,
                                  _stream(stream))
    _check(st, "nt_col_attn_pairbias")


def nt_segment_reduce(op: int, splits_d, v, out, status_d=None, stream=None):
    G, Cc, rows = int(splits_d.shape[0]) - 1, int(v.shape[1]), int(v.shape[0])
    st = lib.nt_segment_reduce(dtype_code(v.dtype), op, Cc, G, rows, _ptr(splits_d), _ptr(v) if rows else None,
                               _ptr(out), _ptr(status_d), _stream(stream))
    _check(st, "nt_segment_reduce")


def nt_transition_workspace_bytes(dtype, c: int, hidden: int, rows: int) -> int:
    return int(lib.nt_transition_workspace_bytes(dtype_code(dtype), c, hidden, rows))


def nt_pair_transition(W: dict, eps: float, z, workspace, status=None, stream=None):
    """z [rows, c] in place; W holds device tensors ln_gamma, ln_beta, W_a, W_b [hidden, c], W_2 [c, hidden]."""
    w = nt_transition_weights(*[_ptr(W[k]) for k in ("ln_gamma", "ln_beta", "W_a", "W_b", "W_2")])
    st = lib.nt_pair_transition(dtype_code(z.dtype), int(z.shape[1]), int(W["W_a"].shape[0]), int(z.shape[0]),
                                C.byref(w), eps, _ptr(z), _ptr(workspace), workspace.nbytes,
                                _ptr(status), _stream(stream))
    _check(st, "nt_pair_transition")


def nt_token_update(m, W_r, x, stream=None):
    st = lib.nt_token_update(dtype_code(x.dtype), int(W_r.shape[0]), int(W_r.shape[1]), int(x.shape[0]),
                             _ptr(m), _ptr(W_r), _ptr(x), _stream(stream))
    _check(st, "nt_token_update")


def nt_launch_count() -> int:
    return int(lib.nt_launch_count())


def nt_debug_expire_wait(status, limit_clocks: int, observed=None, stream=None):
    """One tiny launch whose only wait runs out after limit_clocks SM clocks (testing aid for the timeout path)."""
    st = lib.nt_debug_expire_wait(_ptr(status), int(limit_clocks), _ptr(observed), _stream(stream))
    _check(st, "nt_debug_expire_wait")


NT_PREPARED_WEIGHTS_BYTES = 1 << 20


def nt_prepare_trimul_weights(W: dict, out, stream=None):
    """Folds the LayerNorm parameters into the triangle-update weights once; put `out` into W["prepared"] afterwards."""
    c_h, c_z = int(W["W_ap"].shape[0]), int(W["W_ap"].shape[1])
    w = nt_trimul_weights(*[None if n == "prepared" else _ptr(W[n]) for n, _ in nt_trimul_weights._fields_])
    st = lib.nt_prepare_trimul_weights(dtype_code(W["W_ap"].dtype), c_z, c_h, C.byref(w), _ptr(out),
                                       out.numel() * out.element_size(), _stream(stream))
    _check(st, "nt_prepare_trimul_weights")


def nt_prepare_attn_weights(W: dict, H: int, d: int, out, stream=None):
    """Folds the LayerNorm parameters into the attention weights once; put `out` into W["prepared"] afterwards."""
    c = int(W["W_q"].shape[1])
    w = nt_attn_weights(*[None if n == "prepared" else _ptr(W.get(n)) for n, _ in nt_attn_weights._fields_])
    st = lib.nt_prepare_attn_weights(dtype_code(W["W_q"].dtype), c, H, d, C.byref(w), _ptr(out),
                                     out.numel() * out.element_size(), _stream(stream))
    _check(st, "nt_prepare_attn_weights")


def nt_bench_exp_rate(variant: int, iters: int, blocks: int, sink, clocks, stream=None):
    """Exponential-rate microbenchmark: clocks[block] receives the SM clocks of `iters` rounds of 8 exponentials per thread."""
    st = lib.nt_bench_exp_rate(int(variant), int(iters), int(blocks), _ptr(sink), _ptr(clocks), _stream(stream))
    _check(st, "nt_bench_exp_rate")


def nt_debug_bounds_report(reset: bool = False):
    """(violations, site, index) recorded by the checked build; raises NtError(NT_ERR_UNSUPPORTED) in the normal build."""
    out = (C.c_int32 * 4)()
    _check(lib.nt_debug_bounds_report(out, 1 if reset else 0), "nt_debug_bounds_report")
    return int(out[0]), int(out[1]), (int(out[3]) << 32) | (int(out[2]) & 0xFFFFFFFF)


def nt_debug_attn_drop(blocks: int) -> int:
    return int(lib.nt_debug_attn_drop(int(blocks)))


def nt_attn_core_mode(mode: int) -> int:
    return int(lib.nt_attn_core_mode(int(mode)))


def nt_force_generic(on: bool) -> bool:
    return bool(lib.nt_force_generic(1 if on else 0))


def nt_profile_begin():
    lib.nt_profile_begin()


def nt_profile_end(max_entries: int = 256) -> dict:
    """{kernel name: (total milliseconds, launches)} since nt_profile_begin()."""
    names = C.create_string_buffer(64 * max_entries)
    ms = (C.c_float * max_entries)()
    cnt = (C.c_int64 * max_entries)()
    n = lib.nt_profile_end(C.addressof(names), len(names), C.addressof(ms), C.addressof(cnt), max_entries)
    keys = names.value.decode().split("\n")[:n]
    return {k: (float(ms[i]), int(cnt[i])) for i, k in enumerate(keys)}
