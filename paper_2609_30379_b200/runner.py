"""Sequencing of the library calls for one block / a stack of blocks (the call a user makes).

Only orchestration lives here: buffers come from torch, every arithmetic step is a call into
libnested_pair through ``binding``.  One block (all asynchronous on one stream):
    nt_pair_broadcast -> nt_tri_mul_out -> nt_row_attn_pairbias -> nt_segment_reduce -> nt_token_update
Stacked blocks rebuild the pair state from the tokens the previous block returned and reuse the
same ``z`` and workspace buffers, so peak memory is one block's.
"""
from __future__ import annotations

from typing import List, Optional

import numpy as np
import torch

from . import binding as nt
from .workloads import Config

LN_EPS = 1e-5


def torch_dtype(cfg_dtype: str) -> torch.dtype:
    return torch.float32 if cfg_dtype == "f32" else torch.bfloat16


def to_device(arr: Optional[np.ndarray], dtype: torch.dtype, device="cuda") -> Optional[torch.Tensor]:
    if arr is None:
        return None
    return torch.from_numpy(np.ascontiguousarray(arr)).to(device=device, dtype=dtype).contiguous()


def upload_weights(blocks: List[dict], dtype: torch.dtype, device="cuda") -> List[dict]:
    out = []
    for w in blocks:
        if all(isinstance(v, dict) for v in w.values()):
            out.append({k: {kk: to_device(vv, dtype, device) for kk, vv in v.items()} for k, v in w.items()})
        else:
            out.append({k: to_device(v, dtype, device) for k, v in w.items()})
    return out


class PairStack:
    """Device state for running a configuration's stacked blocks on one batch layout."""

    def __init__(self, cfg: Config, lengths, weights_host: List[dict], device="cuda", fused_mean=True, prepare_weights=True):
        self.cfg = cfg
        self.fused_mean = fused_mean   # nt_row_attn_pairbias_mean instead of attention + nt_segment_reduce
        self.dtype = torch_dtype(cfg.dtype)
        self.device = torch.device(device)
        self.L = nt.Layout(lengths, device=device)
        self.W = upload_weights(weights_host, self.dtype, device)
        dt = nt.dtype_code(self.dtype)
        dims = (cfg.c_s, cfg.c_z, cfg.c_h, cfg.H, cfg.d)
        if cfg.kind == "pair":
            nbytes = nt.nt_workspace_bytes(nt.NT_OP_BLOCK, dt, nt.NT_ORDER_PAIR_IJC, self.L.lengths_h, dims)
            self.z = torch.empty((self.L.T2, cfg.c_z), dtype=self.dtype, device=self.device)
            self.m = torch.empty((self.L.T1, cfg.c_z), dtype=self.dtype, device=self.device)
        else:
            nbytes = nt.nt_workspace_bytes(nt.NT_OP_ROW_ATTN, dt, nt.NT_ORDER_TOKEN_NC, self.L.lengths_h, dims)
            self.z = None
            self.pooled = torch.empty((self.L.B, cfg.c_z), dtype=self.dtype, device=self.device)
        self.workspace = torch.empty(max(nbytes, 256), dtype=torch.uint8, device=self.device)
        if prepare_weights and cfg.kind == "pair" and self.dtype == torch.bfloat16:
            self.prepare_weights()

    def prepare_weights(self):
        """Folds the LayerNorm parameters into the projection weights of every block once (they are constant across
        steps), so that the calls of a step launch no weight preparation.  Shapes the tensor-core stages do not take
        are left as they are (the calls then prepare, or do not need, their own)."""
        for w in self.W:
            for key, fn in (("trimul", lambda W, o: nt.nt_prepare_trimul_weights(W, o)),
                            ("attn", lambda W, o: nt.nt_prepare_attn_weights(W, self.cfg.H, self.cfg.d, o))):
                if key not in w or w[key].get("prepared") is not None:
                    continue
                buf = torch.empty(nt.NT_PREPARED_WEIGHTS_BYTES, dtype=torch.uint8, device=self.device)
                try:
                    fn(w[key], buf)
                except nt.NtError:
                    continue
                w[key]["prepared"] = buf

    # one block, in place on x; z is rebuilt from x
    def block(self, x: torch.Tensor, w: dict, stream=None, accumulate=False):
        cfg, L = self.cfg, self.L
        b = w["broadcast"]
        bc = nt.nt_pair_broadcast_add if accumulate else nt.nt_pair_broadcast
        bc(L, x, b["W_a"], b["W_b"], b["ln_gamma"], b["ln_beta"], LN_EPS, self.z, self.workspace, stream)
        nt.nt_tri_mul_out(L, w["trimul"], LN_EPS, self.z, self.workspace, stream)
        if self.fused_mean:     # attention and the mean over j in one call
            nt.nt_row_attn_pairbias_mean(L, w["attn"], cfg.H, cfg.d, LN_EPS, self.z, self.m, self.workspace, stream)
        else:
            nt.nt_row_attn_pairbias(L, nt.NT_ORDER_PAIR_IJC, w["attn"], cfg.H, cfg.d, LN_EPS, self.z, self.workspace, stream)
            nt.nt_segment_reduce(nt.NT_REDUCE_MEAN, L.row_splits, self.z, self.m, L.status, stream)
        nt.nt_token_update(self.m, w["reduce"]["W_r"], x, stream)

    def capture(self, x: torch.Tensor, persistent=False):
        """Captures forward(x) in a CUDA graph and returns it; graph.replay() reruns every block on the same buffers
        (x is updated in place each time).  Possible because no library call allocates or synchronises; valid for the
        lengths this stack was built with, whose offsets travel by value in the kernel arguments.  Run forward(x) at
        least once before capturing (first calls set kernel attributes)."""
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            self.forward(x, persistent=persistent)
        return graph

    def forward_cached(self, x: torch.Tensor):
        """forward(x) through a graph captured the first time this stack sees the current lengths and this x buffer,
        and replayed afterwards: the kernel arguments carry the batch's offsets by value, so a captured step is valid
        for one length signature; another signature (Layout.rebuild with other lengths) captures again."""
        key = (self.L.lengths_h.tobytes(), x.data_ptr())
        cache = self.__dict__.setdefault("_graphs", {})
        if key not in cache:
            keep = x.clone()
            self.forward(x)                    # first calls set kernel attributes; not captured
            x.copy_(keep)
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                cache[key] = self.capture(x)   # capture does not execute
            torch.cuda.current_stream().wait_stream(side)
        cache[key].replay()
        return (x, self.z) if self.cfg.kind == "pair" else (x, self.pooled)

    def forward(self, x: torch.Tensor, stream=None, persistent=False):
        """Runs every block in place on ``x`` [T1, c_s]; returns (x, z) for pair configs or
        (x, pooled) for the token-only configuration.  persistent=True keeps the pair state as a stream of its
        own: from the second block on the broadcast is accumulated onto it instead of replacing it."""
        if self.cfg.kind == "pair":
            for n, w in enumerate(self.W):
                self.block(x, w, stream, accumulate=persistent and n > 0)
            return x, self.z
        for w in self.W:
            nt.nt_row_attn_pairbias(self.L, nt.NT_ORDER_TOKEN_NC, w, self.cfg.H, self.cfg.d, LN_EPS, x,
                                    self.workspace, stream)
        nt.nt_segment_reduce(nt.NT_REDUCE_MEAN, self.L.tok_off, x, self.pooled, self.L.status, stream)
        return x, self.pooled
