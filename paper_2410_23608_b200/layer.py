"""One pre-norm transformer block around SPA: the device buffers, handed to the library's two layer calls.

out = y1 + FFN(LN2(y1)),  y1 = x + scatter(SPA(LN1(x)))  (paper Sec. 3.2: selected tokens go through attention,
the others are passed straight on to the feed-forward network).  `SpaLayer` owns the buffers; the order
of the kernels lives in the library, as for `SpaBlock`.
"""
from __future__ import annotations

import ctypes

import torch

from . import binding as L
from .block import SpaBlock


class SpaLayer:
    def __init__(self, B: int, N: int, C: int, H: int, dtype: str, hidden: int | None = None, tau: float = 0.0,
                 eps: float = 1e-5, flags: int = 0, device: str = "cuda"):
        self.B, self.N, self.C, self.H = B, N, C, H
        self.hidden = 4 * C if hidden is None else hidden
        self.eps = eps
        # the attention part adds its result to the residual stream: SPA_FLAG_RESIDUAL
        self.blk = SpaBlock(B, N, C, H, dtype, tau=tau, flags=flags | L.SPA_FLAG_RESIDUAL, device=device)
        self.p = self.blk.p
        dev = torch.device(device)
        T = self.blk.tdtype
        rows = max(B * N, 1)
        e = lambda *s, dt=T: torch.empty(*s, dtype=dt, device=dev)
        self.cu_all = (torch.arange(B + 1, dtype=torch.int32, device=dev) * N).contiguous()  # every token is a row
        self.z, self.y1, self.t, self.out = e(B, N, C), e(B, N, C), e(B, N, C), e(B, N, C)
        self.u, self.h = e(rows, self.hidden), e(rows, self.hidden)
        self.m1, self.r1, self.m2, self.r2 = (e(rows, dt=torch.float32) for _ in range(4))
        self.dh, self.dt, self.dy1, self.dX = e(rows, self.hidden), e(B, N, C), e(B, N, C), e(B, N, C)
        f = lambda *s: torch.empty(*s, dtype=torch.float32, device=dev)
        self.dW1, self.db1, self.dW2, self.db2 = f(self.hidden, C), f(self.hidden), f(C, self.hidden), f(C)
        self.dg1, self.dbe1, self.dg2, self.dbe2 = f(C), f(C), f(C), f(C)
        # one area for the caller's stream, one for the weight gradients on the library's second stream
        need = (max(L.spa_layer_workspace_bytes(self.p, self.hidden, side), 256) for side in (False, True))
        self.workspace, self.workspace_side = (torch.empty(n, dtype=torch.uint8, device=dev) for n in need)
        self.blk._bufs.overlap = self.blk._overlap  # the weight gradients on the library's second stream
        self._lib = L.lib()
        own = ("cu_all", "z", "y1", "t", "out", "u", "h", "m1", "r1", "m2", "r2", "dh", "dt", "dy1", "dX", "dW1", "db1", "dW2", "db2",
               "dg1", "dbe1", "dg2", "dbe2", "workspace", "workspace_side")
        self._bufs = L.SpaLayerBuffers(blk=ctypes.pointer(self.blk._bufs), hidden=self.hidden, eps=eps,
                                       **{k: L._ptr(getattr(self, k)) for k in own})
        self._args = (ctypes.byref(self.p), ctypes.byref(self._bufs))

    def forward(self, x, prm):
        """prm: dict of device tensors g1, be1, w_g, W_qkv, b_qkv, W_o, b_o, g2, be2, W1, b1, W2, b2 and float b_g."""
        ptr, l, b = L._ptr, self._bufs, self.blk._bufs
        self._keep = (x, *prm.values())     # the enqueued work and the backward pass read them
        l.x, b.b_g = ptr(x), float(prm["b_g"])
        for k in ("g1", "be1", "g2", "be2", "W1", "b1", "W2", "b2"):
            setattr(l, k, ptr(prm[k]))
        for k in ("w_g", "W_qkv", "b_qkv", "W_o", "b_o"):
            setattr(b, k, ptr(prm[k]))
        L._check(self._lib.spa_layer_fwd(*self._args, L.current_stream_handle()), "spa_layer_fwd")
        return self.out

    def backward(self, d_out):
        """Gradient to x (returned) and to every parameter but the gate's (dW*, db*, dg*, dbe*, and the SPA block's)."""
        self._keep_d = d_out
        self._bufs.d_out = L._ptr(d_out)
        L._check(self._lib.spa_layer_bwd(*self._args, L.current_stream_handle()), "spa_layer_bwd")
        return self.dX

    def read_status(self) -> int:
        return self.blk.read_status()
