"""Scratch of the transformer block's backward pass: what spa_layer_workspace_bytes says is enough, and is no more than it takes."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,C,H,dtype,flag", [
    (32, 256, 768, 12, "bf16", ""), (2, 50, 192, 3, "bf16", ""), (3, 61, 256, 4, "f32", ""),
    (4, 196, 384, 6, "bf16", "SPA_FLAG_NO_CTA_PAIRS"), (2, 50, 128, 2, "bf16", "SPA_FLAG_SIMT_ONLY"),
])
def test_layer_workspace(B, N, C, H, dtype, flag):
    from paper_2410_23608_b200 import binding as L
    from paper_2410_23608_b200.layer import SpaLayer
    T = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(N)
    rnd = lambda *s, std=1.0: (torch.randn(*s, generator=g, device="cuda") * std).to(T)
    F, c = 4 * C, C ** -0.5
    prm = dict(g1=rnd(C), be1=rnd(C), w_g=rnd(C, std=c), b_g=0.1, W_qkv=rnd(3 * C, C, std=c), b_qkv=rnd(3 * C), W_o=rnd(C, C, std=c),
               b_o=rnd(C), g2=rnd(C), be2=rnd(C), W1=rnd(F, C, std=c), b1=rnd(F), W2=rnd(C, F, std=F ** -0.5), b2=rnd(C))
    x, d_out = rnd(B, N, C), rnd(B, N, C)
    lay = SpaLayer(B, N, C, H, dtype, flags=getattr(L, flag) if flag else 0)
    # the weight gradients' partial sums are a few copies of the widest layer, not 32
    assert lay.workspace.numel() + lay.workspace_side.numel() <= 8 * F * C * 4 + (16 << 20)
    need = [L.spa_layer_workspace_bytes(lay.p, F, side) for side in (False, True)]
    names = ("dX", "dW1", "db1", "dW2", "db2", "dg1", "dbe1", "dg2", "dbe2")

    def run():
        lay.forward(x, prm)
        lay.backward(d_out)
        torch.cuda.synchronize()
        assert lay.read_status() == 0
        return [getattr(lay, k).clone() for k in names] + [lay.blk.dW_qkv.clone(), lay.blk.db_qkv.clone(), lay.blk.dW_o.clone()]

    want = run()
    for sizes in (need, [max(max(need), 1)]):       # two areas and the second stream; one area
        area = [torch.full((n + 4096,), 0xA5, dtype=torch.uint8, device="cuda") for n in sizes]
        lay._bufs.workspace, lay._bufs.workspace_side = L._ptr(area[0]), (L._ptr(area[1]) if len(area) > 1 else None)
        for got, ref in zip(run(), want):
            assert torch.equal(got, ref)
        assert all(bool((a[n:] == 0xA5).all()) for a, n in zip(area, sizes))
