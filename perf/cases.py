"""The work that users of this package have it do, as measurable cases.

A case is one call pattern of the public modules (`SpaBlock`, `SpaLayer`) at one size:

  module     "block": one Select-and-Pack-Attention block; "layer": the pre-norm transformer block around it
  mode       "forward" (inference) or "train" (forward and backward)
  dtype      "bf16" or "f32"
  B, rows, cols, C, H      images, token grid, channels, heads (C / H is 32 or 64)
  keep_lo, keep_hi         the images' fractions of selected tokens, spread evenly over this range
  container                0, or the length L of the paper's containers (attention stays inside each container)
  shift                    0, or the cyclic shift of the feature map under which the tokens are packed
  trainable                True: Eq. 5 scaling, up-scale scores and the selection loss; the gradient reaches the gate

Sizes are those of the five workloads (`spa_workloads/configs.py`), of single images and small batches as they occur in
inference, and of grids that no tile divides.  Inputs follow the recipe of `spa_workloads/generate.py`, made on the
GPU: contiguous regions of tokens carry an offset along the gate's weight vector, every gate logit keeps a distance from
the threshold, so the selection (and with it the amount of work) does not depend on rounding.  The number of selected
tokens of a case is fixed; the seed decides which images and which regions hold them, and every value.
"""
from __future__ import annotations

import math

import torch

from paper_2410_23608_b200 import binding as L
from paper_2410_23608_b200.block import SpaBlock
from paper_2410_23608_b200.layer import SpaLayer

ALPHA = 0.5      # weight of the selection loss
OFFSET = 6.0     # length of the offset that selected tokens carry along the gate's weight vector
HIDDEN = 4       # feed-forward width of the layer, in units of C


def _case(name, module, mode, dtype, B, rows, cols, C, H, keep_lo, keep_hi, container=0, shift=0, trainable=False):
    c = dict(module=module, mode=mode, dtype=dtype, B=B, rows=rows, cols=cols, C=C, H=H, keep_lo=keep_lo,
             keep_hi=keep_hi, container=container, shift=shift, trainable=trainable)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one photo through a ViT-S/16 block while a user waits: launches and host work are all there is
        _case("one_image", "block", "forward", "bf16", 1, 14, 14, 384, 6, 0.35, 0.65),
        # the smallest workload: a training step in fp32, as in a first experiment or a numerical check
        _case("tiny_f32_train", "block", "train", "f32", 4, 14, 14, 96, 3, 0.10, 0.50),
        # fp32 inference at an ordinary width, where bf16 is not wanted
        _case("vit_s_f32", "block", "forward", "f32", 16, 14, 14, 384, 6, 0.20, 0.80),
        # a detector on one camera frame of an odd size: few images, long segments
        _case("one_frame", "block", "forward", "bf16", 1, 47, 83, 256, 8, 0.10, 0.40),
        # classification training, small model
        _case("vit_s16_train", "block", "train", "bf16", 64, 14, 14, 384, 6, 0.20, 0.80),
        # detection training: long segments, head dimension 32
        _case("detection_train", "block", "train", "bf16", 16, 50, 84, 256, 8, 0.05, 0.40),
        # large images: half of them nearly empty, half nearly full
        _case("vit_b16_384_train", "block", "train", "bf16", 32, 24, 24, 768, 12, 0.10, 0.90),
        # classification inference in a large batch
        _case("vit_b_infer", "block", "forward", "bf16", 128, 14, 14, 768, 12, 0.01, 0.60),
        # the paper's own batching on the detection grid: containers of 7 x 7 tokens, every second block shifted
        _case("containers_train", "block", "train", "bf16", 16, 50, 84, 256, 8, 0.05, 0.40, container=49, shift=3),
        # supervised, multi-scale selection: the gate is trained with the block; a grid that no tile divides
        _case("gate_train", "block", "train", "bf16", 24, 15, 21, 512, 8, 0.15, 0.75, trainable=True),
        # a whole transformer block, inference on a small batch
        _case("layer_infer", "layer", "forward", "bf16", 8, 14, 14, 384, 6, 0.20, 0.80),
        # a whole transformer block, training
        _case("layer_train", "layer", "train", "bf16", 32, 16, 16, 768, 12, 0.10, 0.90),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Single images to batches of 128, grids from 7 x 7 to detection size, narrow to ViT-L width, in the proportions in
    which the call patterns occur: plain blocks mostly, bf16 mostly."""
    kind = rng.choices(("forward", "train", "containers", "gate", "layer_forward", "layer_train"),
                       weights=(30, 30, 12, 12, 8, 8))[0]
    dtype = "f32" if rng.random() < 1 / 6 else "bf16"
    module = "layer" if kind.startswith("layer") else "block"
    mode = "forward" if kind in ("forward", "layer_forward") else "train"
    if kind == "containers" and rng.random() < 0.3:
        mode = "forward"
    d = rng.choice((32, 64))
    width = 512 if dtype == "f32" else 1024
    H = max(64 // d, min(width // d, _log_int(rng, 3, 16)))
    lo = rng.uniform(0.01, 0.4)
    hi = min(1.0, lo + rng.uniform(0.05, 0.8))
    container = rng.choice((49, 64)) if kind == "containers" else 0
    shift = rng.choice((0, 3)) if kind == "containers" else 0
    while True:
        side = _log_int(rng, 7, 60)
        rows, cols = side, max(7, int(round(side * rng.uniform(0.8, 1.7))))
        B = _log_int(rng, 1, 128)
        c = _case("", module, mode, dtype, B, rows, cols, H * d, H, round(lo, 3), round(hi, 3), container, shift, kind == "gate")
        if rows * cols <= 4200 and _size(c) <= _SIZE_MAX[dtype] and _cost(c) <= _COST_MAX:
            return c


def _size(c):
    return c["B"] * c["rows"] * c["cols"] * c["C"]


def _cost(c):
    """Rough time of a pass in seconds at this package's own rates, to keep drawn cases within the listed ones."""
    w = work(c)
    return w["bytes"] / 3e12 + w["flops"] / (2e13 if c["dtype"] == "f32" else 4e14)


def _counts(c):
    """Selected tokens of each image, in the order before the seed permutes the images."""
    B, N = c["B"], c["rows"] * c["cols"]
    return [max(1, min(N, int(round(N * (c["keep_lo"] + (c["keep_hi"] - c["keep_lo"]) * (b + 0.5) / B))))) for b in range(B)]


def _tokens(gen, c, dev):
    """bool [B, N]: per image the tokens nearest to one to four random centres, as many as _counts says."""
    B, R, K, N = c["B"], c["rows"], c["cols"], c["rows"] * c["cols"]
    n = torch.tensor(_counts(c), device=dev)[torch.randperm(B, generator=gen, device=dev)]
    cy = torch.rand(B, 4, 1, generator=gen, device=dev) * R
    cx = torch.rand(B, 4, 1, generator=gen, device=dev) * K
    size = 0.5 + 0.5 * torch.rand(B, 4, 1, generator=gen, device=dev)
    off = torch.arange(4, device=dev)[None, :, None] > torch.randint(0, 4, (B, 1, 1), generator=gen, device=dev)
    yy = (torch.arange(N, device=dev) // K + 0.5)[None, None]
    xx = (torch.arange(N, device=dev) % K + 0.5)[None, None]
    dist = torch.where(off, torch.inf, ((yy - cy) ** 2 + (xx - cx) ** 2).sqrt() / size).amin(1)
    rank = dist.argsort(1).argsort(1)
    return rank < n[:, None]


def prepare(case, seed):
    c, dev = dict(case), "cuda"
    B, N, C, H = c["B"], c["rows"] * c["cols"], c["C"], c["H"]
    T = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))

    def normal(*shape, std=1.0, mean=0.0):
        return torch.randn(*shape, generator=gen, device=dev).mul_(std).add_(mean).to(T)

    sel = _tokens(gen, c, dev)
    w_g = normal(C, std=C ** -0.5)
    wn = w_g.float().norm()
    u = w_g.float() / wn
    # N(0, 1) values whose part along the gate's weights is cut off at 2.5, plus the offset on the selected tokens
    x = torch.randn(B, N, C, generator=gen, device=dev)
    along = x @ u
    lift = along.clamp(-2.5, 2.5) - along
    s = dict(case=c, sel=sel, w_g=w_g)
    if c["module"] == "layer":
        # LayerNorm rescales a token by its own length, so both kinds of token carry half of the offset
        x += (lift + (sel.float() - 0.5) * OFFSET)[:, :, None] * u
        b_g = 0.0
    else:
        x += (lift + sel.float() * OFFSET)[:, :, None] * u
        b_g = -0.5 * OFFSET * float(wn)
    s["x"], s["b_g"] = x.to(T), b_g
    del x
    s["W_qkv"], s["b_qkv"] = normal(3 * C, C, std=C ** -0.5), normal(3 * C, std=0.02)
    s["W_o"], s["b_o"] = normal(C, C, std=C ** -0.5), normal(C, std=0.02)
    if c["mode"] == "train":
        s["dY"] = normal(B, N, C)
    if c["module"] == "layer":
        F = HIDDEN * C
        s["prm"] = dict(g1=normal(C, std=0.05, mean=1.0), be1=torch.zeros(C, dtype=T, device=dev), w_g=w_g, b_g=b_g,
                        W_qkv=s["W_qkv"], b_qkv=s["b_qkv"], W_o=s["W_o"], b_o=s["b_o"], g2=normal(C, std=0.05, mean=1.0),
                        be2=normal(C, std=0.02), W1=normal(F, C, std=C ** -0.5), b1=normal(F, std=0.02),
                        W2=normal(C, F, std=F ** -0.5), b2=normal(C, std=0.02))
        s["mod"] = SpaLayer(B, N, C, H, c["dtype"])
        return s
    flags = 0
    if c["trainable"]:
        flags = L.SPA_FLAG_GATE_SCALE | L.SPA_FLAG_RESIDUAL
        # scores of the finer stage (a grid twice as dense) agree with the selection; one label in ten does not
        fine = sel.view(B, c["rows"], c["cols"]).repeat_interleave(2, 1).repeat_interleave(2, 2).float()
        noise = torch.randn(fine.shape, generator=gen, device=dev).clamp_(-1.5, 1.5)
        s["scores_fine"] = ((fine - 0.5) * OFFSET + noise).contiguous()
        s["s_up"] = torch.empty(B * N, device=dev)
        flip = torch.rand(B, N, generator=gen, device=dev) < 0.1
        s["labels"] = (sel ^ flip).to(torch.uint8).contiguous()
    if c["shift"]:
        grid = torch.arange(N, dtype=torch.int32, device=dev).view(c["rows"], c["cols"])
        s["order"] = grid.roll((-c["shift"], -c["shift"]), (0, 1)).reshape(-1).contiguous()
    s["mod"] = SpaBlock(B, N, C, H, c["dtype"], flags=flags, backward=c["mode"] == "train")
    return s


def run(state):
    c, m = state["case"], state["mod"]
    if c["module"] == "layer":
        out = {"y": m.forward(state["x"], state["prm"])}
        if c["mode"] == "train":
            out["dX"] = m.backward(state["dY"])
            for k in ("dW1", "db1", "dW2", "db2", "dg1", "dbe1", "dg2", "dbe2"):
                out[k] = getattr(m, k)
            for k in ("dW_qkv", "db_qkv", "dW_o", "db_o"):
                out[k] = getattr(m.blk, k)
        return out
    s_up = None
    if c["trainable"]:
        s_up = state["s_up"]
        L.spa_score_pool(state["scores_fine"], c["B"], c["rows"], c["cols"], s_up)
    y = m.forward(state["x"], state["w_g"], state["b_g"], state["W_qkv"], state["b_qkv"], state["W_o"], state["b_o"],
                  s_up=s_up, order=state.get("order"), container_len=c["container"])
    out = {"y": y, "mask": m.mask, "scores": m.scores, "cu_seqlens": m.cu}
    if c["mode"] == "train":
        keys = ("dW_qkv", "db_qkv", "dW_o", "db_o")
        if c["trainable"]:
            out["dX"] = m.backward_trainable(state["dY"], state["x"], state["w_g"], labels=state["labels"], alpha=ALPHA, s_up=s_up)
            keys += ("ds", "ds_up", "dw_g", "db_g", "loss")
        else:
            out["dX"] = m.backward(state["dY"])
        for k in keys:
            out[k] = getattr(m, k)
    return out


def work(case):
    """Inputs once, outputs once; two operations per multiply-add of Eq. 9's terms (attention's backward is five products
    of the size of one of the forward's two: the probabilities are made again), and of the feed-forward network."""
    c = case
    B, N, C, L_ = c["B"], c["rows"] * c["cols"], c["C"], c["container"]
    es = 4 if c["dtype"] == "f32" else 2
    n = _counts(c)
    Np = sum(n)
    pairs = sum(k * k for k in n) if not L_ else sum((k // L_) * L_ * L_ + (k % L_) ** 2 for k in n)
    train, layer = c["mode"] == "train", c["module"] == "layer"
    weights = 4 * C * C + (2 * HIDDEN * C * C if layer else 0)
    flops = 2 * B * N * C + 8 * Np * C * C + 4 * C * pairs
    nbytes = 2 * B * N * C * es + weights * es
    if layer:
        flops += 4 * B * N * C * HIDDEN * C
    if train:
        flops += 16 * Np * C * C + 10 * C * pairs + (8 * B * N * C * HIDDEN * C if layer else 0)
        nbytes += 2 * B * N * C * es + 4 * weights
    if c["trainable"]:
        flops += 4 * B * N * C
        nbytes += 4 * 4 * B * N + 3 * 4 * B * N
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # fp32: sums of a few hundred to a few thousand terms in another order; bf16: results and intermediates rounded
    # to 8 bits, whose roundings differ between two correct kernels
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2}


_COST_MAX = max(_cost(c) for c in listed())
_SIZE_MAX = {"bf16": max(_size(c) for c in listed()), "f32": 2 * max(_size(c) for c in listed() if c["dtype"] == "f32")}
