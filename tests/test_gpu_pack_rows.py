"""Packing and the transpose of the unpacking at the edges of their batches: rows of 4 to 128 chunks, masks of one load per
thread and of many, tiles of few and of many selected rows."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,C,dtype,keep,flag", [
    (1, 1, 32, "bf16", 1.0, 0),             # one row of four chunks
    (1, 16 * 256, 32, "bf16", 0.5, 0),      # as many mask chunks as threads
    (1, 16 * 256 + 33, 96, "f32", 1.0, 0),  # and more; everything selected
    (3, 1357, 384, "bf16", 0.3, "RESIDUAL"),
    (16, 4200, 64, "bf16", 0.9, 0),         # more than one batch of mask loads
    (5, 301, 1024, "bf16", 0.0, 0),         # nothing selected
    (2, 500, 512, "f32", 0.7, "RESIDUAL"),  # 128 chunks a row
    (7, 77, 768, "bf16", 0.6, 0),
])
def test_pack_and_its_transposes_move_rows(B, N, C, dtype, keep, flag):
    from paper_2410_23608_b200 import binding as L
    T = torch.float32 if dtype == "f32" else torch.bfloat16
    flags = getattr(L, "SPA_FLAG_" + flag) if flag else 0
    p = L.make_params(B, N, C, max(C // 32, 1), dtype, B * N, flags)
    g = torch.Generator(device="cuda").manual_seed(B * N + C)
    x, dY = (torch.randn(B * N, C, generator=g, device="cuda").to(T) for _ in range(2))
    mask = (torch.rand(B * N, generator=g, device="cuda") < keep).to(torch.uint8)
    sel = mask.nonzero()[:, 0].int()
    Np = sel.numel()
    e = lambda *s, dt=torch.int32: torch.full(s, 7, device="cuda", dtype=dt)
    xp, idx, inv, cu, status = e(B * N, C, dt=T), e(B * N), e(B * N), e(B + 1), torch.zeros(4, dtype=torch.int32, device="cuda")
    L.spa_select_pack(p, x, mask, None, xp, idx, inv, cu, status)
    assert L.spa_read_status(status) == 0
    assert torch.equal(xp[:Np], x[sel.long()]) and bool((xp[Np:] == 7).all())
    assert torch.equal(idx[:Np], sel) and bool((idx[Np:] == 7).all())
    want = torch.full_like(inv, -1)
    want[sel.long()] = torch.arange(Np, device="cuda", dtype=torch.int32)
    assert torch.equal(inv, want)
    assert cu.tolist() == [0] + mask.view(B, N).sum(1).cumsum(0).tolist()
    for in_place in (False, True):
        d = dY.clone()
        dz, dX = e(B * N, C, dt=T), d if in_place else e(B * N, C, dt=T)
        L.spa_unpack_scatter_bwd(p, d, idx, inv, cu, dz, dX)
        torch.cuda.synchronize()
        assert torch.equal(dz[:Np], dY[sel.long()]) and bool((dz[Np:] == 7).all())
        if in_place:
            assert torch.equal(dX, dY)
        else:
            assert torch.equal(dX[mask == 0], dY[mask == 0])
            assert torch.equal(dX[mask == 1], dY[mask == 1]) if flag else bool((dX[mask == 1] == 7).all())


@pytest.mark.parametrize("rows,C,dtype,keep,flag", [
    (7, 8, "bf16", 0.5, 0),                  # one chunk a row: every chunk of a thread in another row
    (784, 96, "f32", 0.3, 0),                # 24 chunks a row: rows across warps and CTAs
    (301, 8192, "f32", 0.4, "RESIDUAL"),     # 2 048 chunks a row: longer than a CTA's step
    (18944, 256, "bf16", 0.3, 0),            # two chunks a thread: the most
    (18945, 256, "bf16", 0.3, "RESIDUAL"),   # four, and whole rows to a warp where nothing is copied
    (15001, 328, "bf16", 0.6, 0),            # 41 chunks a row: a warp's second pass is partly empty
    (86017, 56, "bf16", 0.2, 0),             # 7 chunks a row
    (42000, 1024, "bf16", 0.1, 0),           # more than one step for a CTA
])
def test_transpose_of_the_unpacking(rows, C, dtype, keep, flag):
    from paper_2410_23608_b200 import binding as L
    T = torch.float32 if dtype == "f32" else torch.bfloat16
    p = L.make_params(1, rows, C, 1, dtype, rows, getattr(L, "SPA_FLAG_" + flag) if flag else 0)
    g = torch.Generator(device="cuda").manual_seed(rows + C)
    dY = torch.randn(rows, C, generator=g, device="cuda").to(T)
    sel = torch.rand(rows, generator=g, device="cuda") < keep
    Np = int(sel.sum())
    for n_valid in (Np, Np - Np // 3):                      # all packed rows, and fewer than the places say
        inv = torch.where(sel, sel.cumsum(0) - 1, -1).int()
        cu = torch.tensor([0, n_valid], dtype=torch.int32, device="cuda")
        taken = sel & (inv < n_valid)
        for target in ("dX", "dY", None):
            d, dz = dY.clone(), torch.full((rows, C), 7, device="cuda", dtype=T)
            dX = torch.full((rows, C), 7, device="cuda", dtype=T) if target == "dX" else d if target else None
            L.spa_unpack_scatter_bwd(p, d, None, inv, cu, dz, dX)
            torch.cuda.synchronize()
            assert torch.equal(dz[:n_valid], dY[taken]) and bool((dz[n_valid:] == 7).all())
            assert torch.equal(d, dY)
            if target == "dX":
                assert torch.equal(dX[~taken], dY[~taken])
                assert torch.equal(dX[taken], dY[taken]) if flag else bool((dX[taken] == 7).all())


@pytest.mark.parametrize("B,N,C,dtype,keep,scaled,shift,short", [
    (3, 50, 8, "bf16", 1.0, False, 0, 0),       # one chunk a row: a thread's next one is 256 rows on
    (7, 1000, 40, "bf16", 0.7, True, 9, 0),     # five chunks a row: 256 is no multiple
    (2, 700, 1016, "f32", 0.9, True, 0, 0),     # 254 chunks
    (2, 700, 1028, "f32", 0.9, True, 5, 0),     # 257: longer than the CTA's step
    (1, 67, 8192, "f32", 0.8, False, 0, 0),     # 2 048 chunks a row
    (64, 196, 192, "bf16", 0.5, False, 0, 100), # rows that do not fit in
    (2, 30000, 16, "bf16", 0.02, False, 0, 0),  # long counts, nearly empty tiles
])
def test_packing_in_batches(B, N, C, dtype, keep, scaled, shift, short):
    from paper_2410_23608_b200 import binding as L
    T = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B * N + C)
    x = torch.randn(B, N, C, generator=g, device="cuda").to(T)
    scores = torch.randn(B, N, generator=g, device="cuda")
    sel = torch.rand(B, N, generator=g, device="cuda") < keep
    # any non-zero byte selects
    mask = torch.where(sel, torch.randint(1, 256, (B, N), generator=g, device="cuda"), 0).to(torch.uint8).contiguous()
    visit = torch.arange(N, device="cuda").roll(-shift)
    tok = (torch.arange(B, device="cuda")[:, None] * N + visit).reshape(-1)
    tok = tok[sel.reshape(-1)[tok]]
    Np = tok.numel()
    cap = Np - short
    p = L.make_params(B, N, C, 1, dtype, cap, L.SPA_FLAG_GATE_SCALE if scaled else 0)
    e = lambda *s, dt=torch.int32: torch.full(s, 7, device="cuda", dtype=dt)
    xp, idx, inv, cu, status = e(cap + 3, C, dt=T), e(cap + 3), e(B * N), e(B + 1), torch.zeros(4, dtype=torch.int32, device="cuda")
    if shift:
        L.spa_select_pack_ordered(p, x, mask, scores, visit.int(), xp, idx, inv, cu, status)
    else:
        L.spa_select_pack(p, x, mask, scores, xp, idx, inv, cu, status)
    assert L.spa_read_status(status) == (L.SPA_ERR_CAPACITY if short else 0)
    tok = tok[:cap]
    want = x.view(-1, C)[tok]
    if scaled:  # 1 / (1 + exp(-s)): the exponential is good to 2 + 1.16 |s| units in the last place, |s| < 6
        ref = (want.double() * scores.view(-1)[tok].double().sigmoid()[:, None])
        assert bool(((xp[:cap].double() - ref).abs() <= (2e-6 if dtype == "f32" else 2 ** -8) * ref.abs()).all())
    else:
        assert torch.equal(xp[:cap], want)
    assert torch.equal(idx[:cap], tok.int()) and bool((xp[cap:] == 7).all()) and bool((idx[cap:] == 7).all())
    place = torch.full((B * N,), -1, device="cuda", dtype=torch.int32)
    place[tok] = torch.arange(cap, device="cuda", dtype=torch.int32)
    assert torch.equal(inv, place)
    assert cu.tolist() == [0] + sel.sum(1).cumsum(0).tolist()
