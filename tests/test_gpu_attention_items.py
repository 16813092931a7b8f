"""Attention forward: how its CTAs come by their work - one item each, drawn in order or as they stand, in launches and in
recorded ones - with offsets in registers, in shared memory or in global memory."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,H,lengths", [
    (64, 1, [1]),                                 # one row
    (64, 12, [577, 58] * 9),                      # items drawn, put in order of length
    (32, 8, [1680] + [0] * 3 + [210] * 40),       # in order; empty segments
    (64, 12, [700] * 5 + [131]),                  # a few more items than CTAs
    (32, 16, [49] * 511),                         # offsets of the first item by one warp: the most
    (64, 8, [49] * 512),                          # and one more; drawn without order
    (32, 4, [5] * 2047),                          # staged offsets: the most
    (64, 4, [5] * 2048 + [300] * 30),             # and one more
    (32, 1, [3] * 70001),                         # more row tiles than are put in order
])
def test_attention_forward_items(d, H, lengths):
    from paper_2410_23608_b200 import binding as L
    C, Np, n_seg = H * d, sum(lengths), len(lengths)
    cap = Np + 70
    g = torch.Generator(device="cuda").manual_seed(Np)
    qkv = torch.randn(cap, 3 * C, generator=g, device="cuda").to(torch.bfloat16)
    qkv[Np:] = float("nan")                       # rows past the last packed one are unspecified
    n = torch.tensor(lengths, device="cuda")
    cu = torch.cat([n.new_zeros(1), n.cumsum(0)]).int()
    p = L.make_params(1, cap, C, H, "bf16", cap)
    ao, lse = torch.empty(cap, C, device="cuda", dtype=torch.bfloat16), torch.empty(H, cap, device="cuda")
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    run = lambda: L.spa_packed_attention_fwd(p, qkv, cu, n_seg, ao, lse, status)
    # reference: segments of equal length together, padded to the longest
    pad = max(lengths)
    row = cu[:-1, None] + torch.arange(pad, device="cuda")
    valid = torch.arange(pad, device="cuda") < n[:, None]
    q, k, v = qkv[torch.where(valid, row, 0)].float().view(n_seg, pad, 3, H, d).permute(2, 0, 3, 1, 4)
    s = (q @ k.transpose(-1, -2) * d ** -0.5).masked_fill(~valid[:, None, None], float("-inf"))
    o = (torch.nan_to_num(s.softmax(-1)) @ v).permute(0, 2, 1, 3).reshape(n_seg, pad, C)[valid]
    ref_lse = s.logsumexp(-1).permute(1, 0, 2)[:, valid]

    def check():
        assert L.spa_read_status(status) == 0
        assert float((ao[:Np].float() - o).abs().max()) < 2e-2 and float((lse[:, :Np] - ref_lse).abs().max()) < 1e-3
        assert bool((ao[Np:] == 7).all()) and bool((lse[:, Np:] == 7).all())
        first = ao.clone()
        ao.fill_(7)
        lse.fill_(7)
        return first

    ao.fill_(7), lse.fill_(7)
    run()
    first = check()
    run()                                         # the counter is back at zero
    assert torch.equal(check(), first)
    graphs = [torch.cuda.CUDAGraph() for _ in range(2)]
    for gr in graphs:
        with torch.cuda.graph(gr):
            run()
    for gr in graphs + graphs:
        gr.replay()
        assert torch.equal(check(), first)
