"""One SPA block: the device buffers, handed to the library's two block calls.

`SpaBlock` owns the buffers of one block (allocated once through PyTorch) and calls `spa_block_fwd` /
`spa_block_bwd` on the current stream.  The order of the kernels, the choice between fused and separate
scatter calls and the second stream for the weight gradients all live in the library; nothing here
computes or sequences.  Nothing synchronises; N_p stays on the device.
"""
from __future__ import annotations

import ctypes
from typing import Optional

import torch

from . import binding as L


class SpaBlock:
    """Buffers for gate -> select/pack -> QKV -> attention -> projection -> unpack (paper Sec. 3.2) and the
    matching backward pass."""

    def __init__(self, B: int, N: int, C: int, H: int, dtype: str, tau: float = 0.0, flags: int = 0,
                 capacity: Optional[int] = None, backward: bool = True, device: str = "cuda",
                 fused: Optional[bool] = None, one_pass: bool = False):
        if not torch.cuda.is_available():
            raise RuntimeError("SpaBlock needs a CUDA device; there is no CPU path")
        self._lib = L.lib()
        self.B, self.N, self.C, self.H = B, N, C, H
        self.tdtype = torch.float32 if dtype == "f32" else torch.bfloat16
        cap = capacity if capacity is not None else max(B * N, 1)
        # fused unpack: the projection and the QKV input gradient scatter their rows to the tokens themselves; False =
        # separate kernels.  `self.fused`: the single calls that do so apply too (tensor-core problems)
        can_fuse = L.spa_fused_scatter_supported(L.make_params(B, N, C, H, dtype, cap, flags, tau))
        if fused and not can_fuse:
            raise ValueError("the fused scatter calls do not apply to this problem (needs bf16 tensor-core sizes)")
        self.fused = can_fuse if fused is None else bool(fused)
        if fused is False:
            flags |= L.SPA_FLAG_UNFUSED
        self.p = L.make_params(B, N, C, H, dtype, cap, flags, tau)
        self.cap = cap
        self._inplace = bool(flags & L.SPA_FLAG_INPLACE)
        dev = torch.device(device)
        T = self.tdtype
        e = lambda *s, dt=T: torch.empty(*s, dtype=dt, device=dev)
        self.scores = e(max(B * N, 1), dt=torch.float32)
        self.mask = e(max(B * N, 1), dt=torch.uint8)
        self.cu = torch.zeros(B + 1, dtype=torch.int32, device=dev)
        self.idx = e(cap, dt=torch.int32)
        self.inv = e(max(B * N, 1), dt=torch.int32)
        self.xp = e(cap, C)
        self.qkv = e(cap, 3 * C)
        self.ao = e(cap, C)
        self.lse = e(H, cap, dt=torch.float32)
        self.z = e(cap, C)
        self.y = e(B, N, C)
        self.status = torch.zeros(4, dtype=torch.int32, device=dev)
        ws = L.spa_workspace_bytes(self.p)
        self.workspace = torch.empty(max(ws, 256), dtype=torch.uint8, device=dev) if ws > 0 else None
        # the weight gradients run on a second stream (owned by the library handle), with a scratch area of their own
        self.workspace_side = torch.empty(max(ws, 256), dtype=torch.uint8, device=dev) if (ws > 0 and backward) else None
        self._overlap = L.spa_overlap_create() if backward else None
        # one_pass: gate, selection and packing as one kernel (measured slower than the two kernels on the five
        # workloads, so off unless asked for); its scratch is zeroed once here, the kernel leaves it zero
        self.one_pass = one_pass and L.spa_gate_select_pack_supported(self.p)
        self.pack_state = (torch.zeros(max(L.spa_pack_state_bytes(self.p), 256), dtype=torch.uint8, device=dev)
                           if self.one_pass else None)
        if backward:
            self.dz = e(cap, C)
            self.dao = e(cap, C)
            self.dqkv = e(cap, 3 * C)
            self.dxp = e(cap, C)
            self.dX = e(B, N, C)
            self.dW_qkv = e(3 * C, C, dt=torch.float32)
            self.db_qkv = e(3 * C, dt=torch.float32)
            self.dW_o = e(C, C, dt=torch.float32)
            self.db_o = e(C, dt=torch.float32)
        self._saved = None            # (W_qkv, W_o) of the last forward()
        self._keep = None             # tensors of the last call that the enqueued work still reads
        self._n_max = {}              # container length -> upper bound of the number of containers
        self.container_seg = None
        self._bufs = self._fixed_buffers(backward)  # segments: the images, unless forward() is given others
        self._args = (ctypes.byref(self.p), ctypes.byref(self._bufs))

    def __del__(self):
        try:
            if getattr(self, "_overlap", None):
                torch.cuda.synchronize()
                L.spa_overlap_destroy(self._overlap)
                self._overlap = None
        except Exception:
            pass

    def _fixed_buffers(self, backward):
        """The block's own buffers as the library's struct, filled once: a call sets only the tensors it is given.
        (Filling all of it anew cost 10 us of the 38 us a forward call of one image spent on the host.)"""
        f = dict(scores=self.scores, mask=self.mask, cu_seqlens=self.cu, idx=self.idx, inv=self.inv, x_packed=self.xp,
                 qkv=self.qkv, attn_out=self.ao, lse=self.lse, z=self.z, workspace=self.workspace, d_status=self.status,
                 pack_state=self.pack_state)
        if backward:
            f.update(dz=self.dz, d_attn_out=self.dao, dqkv=self.dqkv, dx_packed=self.dxp, dW_qkv=self.dW_qkv,
                     db_qkv=self.db_qkv, dW_o=self.dW_o, db_o=self.db_o, workspace_side=self.workspace_side)
        return L.block_buffers(**f)

    # ------------------------------------------------------------------ forward
    def forward(self, x, w_g, b_g: float, W_qkv, b_qkv, W_o, b_o, s_up=None, y=None, order=None, seg_offsets=None,
                container_len: int = 0):
        """`order` (int32 [N] on the device): visiting order of each image's tokens for the packing (a shifted
        feature map); `seg_offsets` (int32, ascending, ending at N_p): attention segments other than the images;
        `container_len` = L > 0: the paper's containers, their cuts built on the device by the library (the segment
        array is owned here).  The backward pass uses the same segments."""
        ptr, b = L._ptr, self._bufs
        y = x if self._inplace else (self.y if y is None else y)
        if container_len > 0:
            n_max = self._n_max.get(container_len)
            if n_max is None:
                n_max = self._n_max[container_len] = L.spa_container_max_segments(self.p, container_len)
            if self.container_seg is None or self.container_seg.numel() != n_max + 1:
                self.container_seg = torch.zeros(n_max + 1, dtype=torch.int32, device=self.cu.device)
            seg_offsets = self.container_seg
        b.container_len = int(container_len)
        if seg_offsets is None:
            b.seg_offsets, b.n_seg = None, self.B
        else:
            b.seg_offsets, b.n_seg = ptr(seg_offsets), int(seg_offsets.numel()) - 1
        self._saved = (W_qkv, W_o)
        self._keep = (x, w_g, W_qkv, b_qkv, W_o, b_o, s_up, order, seg_offsets, y)
        b.x, b.w_g, b.b_g, b.s_up, b.order, b.y = ptr(x), ptr(w_g), float(b_g), ptr(s_up), ptr(order), ptr(y)
        b.W_qkv, b.b_qkv, b.W_o, b.b_o = ptr(W_qkv), ptr(b_qkv), ptr(W_o), ptr(b_o)
        L._check(self._lib.spa_block_fwd(*self._args, L.current_stream_handle()), "spa_block_fwd")
        return y

    # ------------------------------------------------------------------ backward
    def _backward(self, dY, dX, overlap, trainable):
        b = self._bufs
        W_qkv, W_o = self._saved
        b.W_qkv, b.W_o, b.dY, b.dX = L._ptr(W_qkv), L._ptr(W_o), L._ptr(dY), L._ptr(dX)
        b.overlap, b.trainable = overlap, trainable
        L._check(self._lib.spa_block_bwd(*self._args, L.current_stream_handle()), "spa_block_bwd")
        return dX

    def backward(self, dY, dX=None, overlap=True):
        """Gradients for the last forward(): returns dX; parameter gradients land in dW_qkv, db_qkv,
        dW_o, db_o (fp32).  No gradient reaches the gate (hard threshold).  With overlap=True the two
        weight-gradient products run on the library's second stream and are joined before the call returns."""
        return self._backward(dY, self.dX if dX is None else dX, self._overlap if overlap else None, 0)

    def backward_trainable(self, dY, x, w_g, labels=None, alpha: float = 1.0, s_up=None, dX=None):
        """backward() extended by the gradient that reaches the gate (Sec. 3.2 Eq. 4-5, Sec. 3.3 Eq. 10): the
        selection loss alpha * BCE(Sigmoid(scores), labels) when `labels` (uint8 [B, N]) is given, and, under
        SPA_FLAG_GATE_SCALE, the path through the sigmoid scaling of the packed rows.  `s_up` must be the
        tensor given to forward().  Returns dX; also fills dw_g, db_g, ds_up (fp32), ds and loss."""
        dX = self.dX if dX is None else dX
        if not hasattr(self, "ds"):
            dev = self.scores.device
            n = max(self.B * self.N, 1)
            self.ds = torch.empty(n, dtype=torch.float32, device=dev)
            self.ds_up = torch.empty(n, dtype=torch.float32, device=dev)
            self.dw_g = torch.empty(self.C, dtype=torch.float32, device=dev)
            self.db_g = torch.empty(1, dtype=torch.float32, device=dev)
            self.loss = torch.zeros(1, dtype=torch.float32, device=dev)
            self.train_ws = torch.empty(max(L.spa_train_workspace_bytes(self.p), 256), dtype=torch.uint8, device=dev)
            b = self._bufs
            b.ds, b.ds_up, b.dw_g, b.db_g = L._ptr(self.ds), L._ptr(self.ds_up), L._ptr(self.dw_g), L._ptr(self.db_g)
            b.loss, b.train_workspace = L._ptr(self.loss), L._ptr(self.train_ws)
        b = self._bufs
        b.x, b.w_g, b.s_up, b.labels, b.alpha = L._ptr(x), L._ptr(w_g), L._ptr(s_up), L._ptr(labels), float(alpha)
        return self._backward(dY, dX, self._overlap, 1)

    def read_status(self) -> int:
        """Blocking: the device status word (0 = ok)."""
        return L.spa_read_status(self.status)
