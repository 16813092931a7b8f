"""A device-side wait that runs out inside a linear layer's tensor-core kernel: the call ends with SPA_ERR_TIMEOUT, the copies
and products in flight have been waited for, and ordinary calls behind it on the same stream are correct."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# forward and input gradient on CTA pairs, weight gradient on CTA pairs (a last k-block of 5 rows); on single CTAs; on clusters
@pytest.mark.parametrize("rows,n_in,n_out,pairs", [(9221, 768, 2304, True), (2309, 768, 768, False), (5997, 384, 384, True),
                                                   (14411, 256, 768, True)])
def test_short_waits_leave_nothing_in_flight(rows, n_in, n_out, pairs):
    from paper_2410_23608_b200 import binding as L
    g = torch.Generator(device="cuda").manual_seed(rows)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    flags = 0 if pairs else L.SPA_FLAG_NO_CTA_PAIRS
    p, short = (L.make_params(1, 2 * rows, 64, 2, "bf16", 2 * rows, flags=f) for f in (flags, flags | L.SPA_FLAG_SHORT_WAITS))
    cu = torch.tensor([0, rows], dtype=torch.int32, device="cuda")
    a, W, dout = rnd(2 * rows, n_in), rnd(n_out, n_in), rnd(2 * rows, n_out)
    ws = torch.empty(160 << 20, dtype=torch.uint8, device="cuda")

    def calls(p, status):
        out, da = torch.empty(2 * rows, n_out, device="cuda").bfloat16(), torch.empty(2 * rows, n_in, device="cuda").bfloat16()
        dW, db = torch.empty(n_out, n_in, device="cuda"), torch.empty(n_out, device="cuda")
        L.spa_packed_linear(p, a, W, None, n_in, n_out, cu, out, d_status=status[0])
        L.spa_packed_linear_bwd(p, a, W, dout, n_in, n_out, cu, da, None, None, ws, d_status=status[1])
        L.spa_packed_linear_bwd(p, a, W, dout, n_in, n_out, cu, None, dW, db, ws, d_status=status[2])
        return out[:rows], da[:rows], dW, db

    clean, expired = torch.zeros(3, 4, dtype=torch.int32, device="cuda"), torch.zeros(3, 4, dtype=torch.int32, device="cuda")
    want = calls(p, clean)
    for _ in range(10):
        calls(short, expired)
        got = calls(p, clean)                 # right behind, without a synchronisation
        assert all(torch.equal(x, y) for x, y in zip(got, want))
    assert [L.spa_read_status(s) for s in clean] == [0, 0, 0]
    assert [L.spa_read_status(s) for s in expired] == [L.SPA_ERR_TIMEOUT] * 3


# items drawn in order of length; given and drawn, one or two tiles each; one per CTA; two CTAs.  A poll itself waits for a time that the
# hardware sets, about as long as a copy takes: only with many items per CTA is one certain to fail
@pytest.mark.parametrize("d,H,cap,lengths,certain", [(64, 12, 18432, [577, 58] * 9, True), (32, 16, 34000, [49] * 511, True),
                                                     (64, 12, 34000, [700], False), (32, 2, 1 << 18, [100], False)])
def test_short_waits_in_the_attention_backward(d, H, cap, lengths, certain):
    from paper_2410_23608_b200 import binding as L
    C, Np, n_seg = H * d, sum(lengths), len(lengths)
    g = torch.Generator(device="cuda").manual_seed(Np)
    qkv = torch.randn(cap, 3 * C, generator=g, device="cuda").to(torch.bfloat16)
    dao = torch.randn(cap, C, generator=g, device="cuda").to(torch.bfloat16)
    ao, lse = torch.empty(cap, C, device="cuda", dtype=torch.bfloat16), torch.empty(H, cap, device="cuda")
    cu = torch.tensor([0] + lengths, device="cuda").cumsum(0).int()
    p, short = (L.make_params(1, cap, C, H, "bf16", cap, flags=f) for f in (0, L.SPA_FLAG_SHORT_WAITS))
    ws = torch.empty(max(L.spa_workspace_bytes(p), 256), dtype=torch.uint8, device="cuda")
    clean, expired = torch.zeros(4, dtype=torch.int32, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    L.spa_packed_attention_fwd(p, qkv, cu, n_seg, ao, lse, clean)
    out = torch.full((cap, 3 * C), 7.0, device="cuda", dtype=torch.bfloat16)
    run = lambda p, status: L.spa_packed_attention_bwd(p, qkv, ao, lse, dao, cu, n_seg, out, ws, status)
    run(p, clean)
    want = out.clone()
    for _ in range(10):
        run(short, expired)
        assert bool((out[Np:] == 7).all())
        run(p, clean)                         # the same array: its items are counted from zero again
        assert torch.equal(out, want)
    assert L.spa_read_status(clean) == 0
    assert L.spa_read_status(expired) in ((L.SPA_ERR_TIMEOUT,) if certain else (0, L.SPA_ERR_TIMEOUT))
