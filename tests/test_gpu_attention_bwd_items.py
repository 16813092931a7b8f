"""Attention backward in one pipeline per CTA over all its items (attn_bwd_kv.cu, large problems): items given, drawn
and put in order, one tile and many, few offsets and many, and what the other kernels take."""
import pytest
import torch

from tests.gpu_util import assert_close, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,H,cap,lengths", [
    (64, 1, 1 << 18, [1]),                                  # one row, in a capacity that stands for many
    (32, 2, 1 << 18, [129]),                                # two items of two tiles each
    (64, 12, 18432, [577, 58] * 9),                         # in order of length, drawn
    (32, 8, 67200, [1680] + [0] * 3 + [210] * 40),          # empty segments
    (64, 12, 34000, [128] * 40 + [1] * 128 + [256, 384]),   # boundaries on the tiles; items of one tile
    (32, 16, 34000, [49] * 511),                            # the first item by one warp: the most segments
    (64, 12, 34000, [49] * 512),                             # and one more
    (32, 16, 34000, [5] * 2047),                             # offsets in the least shared memory that is asked for
    (64, 8, 80000, [5] * 2048 + [300] * 30),                # and more
    (64, 4, 100000, [8] * 12287),                            # staged offsets: the most
    (32, 4, 100000, [8] * 12288),                            # and one more: the other kernels
    (32, 4, 140000, [3] * 40001),                           # offsets in global memory: the other kernels, many row tiles
    (64, 2, 80000, [300, 700] * 75 + [8]),                  # 512 drawn row tiles: the most that are put in order
    (64, 2, 80000, [300, 700] * 75 + [9]),                  # and one more
    (64, 2, 300, [100, 77, 123]),                           # too small: the other kernels
])
def test_attention_backward_items(d, H, cap, lengths):
    from paper_2410_23608_b200 import binding as L
    C, Np, n_seg = H * d, sum(lengths), len(lengths)
    g = torch.Generator(device="cuda").manual_seed(Np + d)
    qkv = torch.randn(cap, 3 * C, generator=g, device="cuda").to(torch.bfloat16)
    dao = torch.randn(cap, C, generator=g, device="cuda").to(torch.bfloat16)
    ao, lse = torch.empty(cap, C, device="cuda", dtype=torch.bfloat16), torch.empty(H, cap, device="cuda")
    for t in (qkv, dao, ao):
        t[Np:] = float("nan")                               # rows past the last packed one are unspecified
    n = torch.tensor(lengths, device="cuda")
    cu = torch.cat([n.new_zeros(1), n.cumsum(0)]).int()
    p = L.make_params(1, cap, C, H, "bf16", cap)
    ws = torch.empty(max(L.spa_workspace_bytes(p), 256), dtype=torch.uint8, device="cuda")
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    L.spa_packed_attention_fwd(p, qkv, cu, n_seg, ao, lse, status)
    out = torch.full((cap, 3 * C), 7.0, device="cuda", dtype=torch.bfloat16)
    run = lambda: L.spa_packed_attention_bwd(p, qkv, ao, lse, dao, cu, n_seg, out, ws, status)
    # reference: segments padded to the longest, fp32
    pad = max(lengths)
    valid = torch.arange(pad, device="cuda") < n[:, None]
    row = torch.where(valid, cu[:-1, None] + torch.arange(pad, device="cuda"), 0)
    x = qkv[row].float().view(n_seg, pad, 3, H, d).permute(2, 0, 3, 1, 4).contiguous().requires_grad_()
    s = (x[0] @ x[1].transpose(-1, -2) * d ** -0.5).masked_fill(~valid[:, None, None], float("-inf"))
    o = torch.nan_to_num(s.softmax(-1)) @ x[2]
    do = dao[row].float().view(n_seg, pad, H, d).transpose(1, 2) * valid[:, None, :, None]
    o.backward(do)
    ref = host(x.grad.permute(1, 3, 0, 2, 4).reshape(n_seg, pad, 3 * C)[valid])

    def check():
        assert L.spa_read_status(status) == 0
        got = host(out)[:Np]
        for i, name in enumerate(("dQ", "dK", "dV")):
            assert_close(got[:, i * C:(i + 1) * C], ref[:, i * C:(i + 1) * C], "bf16", name, scale_max_abs=True)
        assert bool((out[Np:] == 7).all())
        first = out.clone()
        out.fill_(7)
        return first

    run()
    first = check()
    run()                                                   # the counter is back at zero
    assert torch.equal(check(), first)
    gr = torch.cuda.CUDAGraph()
    with torch.cuda.graph(gr):
        run()
    for _ in range(20):
        gr.replay()
    assert torch.equal(check(), first)


@pytest.mark.parametrize("d,H", [(64, 12), (32, 16)])
@pytest.mark.parametrize("rows", [129, 300, 320, 384])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_what_is_not_finite_stays_with_the_tiles_of_its_image(d, H, rows, bad):
    """dK and dV of 128 packed rows read the images that have rows among them, and no row behind those images."""
    from paper_2410_23608_b200 import binding as L
    C, cap, lengths = H * d, 34000, [rows, 500, 128 * 4 - (rows + 500) % 128, 777]
    Np = sum(lengths)
    g = torch.Generator(device="cuda").manual_seed(rows)
    qkv = torch.randn(cap, 3 * C, generator=g, device="cuda").to(torch.bfloat16)
    dao = torch.randn(cap, C, generator=g, device="cuda").to(torch.bfloat16)
    ao, lse = torch.empty(cap, C, device="cuda", dtype=torch.bfloat16), torch.empty(H, cap, device="cuda")
    cu = torch.tensor([0] + lengths, device="cuda").cumsum(0).int()
    p = L.make_params(1, cap, C, H, "bf16", cap)
    ws = torch.empty(max(L.spa_workspace_bytes(p), 256), dtype=torch.uint8, device="cuda")
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    L.spa_packed_attention_fwd(p, qkv, cu, 4, ao, lse, status)

    def backward():
        out = torch.empty(cap, 3 * C, device="cuda", dtype=torch.bfloat16)
        L.spa_packed_attention_bwd(p, qkv, ao, lse, dao, cu, 4, out, ws, status)
        assert L.spa_read_status(status) == 0
        return out[:Np, C:]

    want = backward()
    bad_rows = slice(rows, rows + 500)                      # the second image
    dao[bad_rows] = bad
    got = backward()
    alone = torch.ones(Np, dtype=torch.bool, device="cuda")
    alone[rows // 128 * 128:(rows + 500 + 127) // 128 * 128] = False
    assert torch.equal(got[alone], want[alone])
    assert not bool(torch.isfinite(got[bad_rows]).any())
