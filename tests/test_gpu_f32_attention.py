"""fp32 attention: what one image holds does not reach another one."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("d", [32, 64])
def test_nonfinite_values_stay_in_their_segment(d, value):
    """Segments of 5 to 150 rows, so that tiles of own and of streamed rows hold several: with infinities or NaN in the rows of
    two of them, the rows of the others come out as without, forward and backward."""
    from paper_2410_23608_b200 import binding as L
    H, cuts = 2, [0, 20, 45, 50, 200, 231, 300]
    C, rows = H * d, cuts[-1]
    g = torch.Generator(device="cuda").manual_seed(d)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    p = L.make_params(1, rows, C, H, "f32", rows)
    seg = torch.tensor(cuts, dtype=torch.int32, device="cuda")
    qkv, dao = rnd(rows, 3 * C), rnd(rows, C)
    bad = torch.zeros(rows, dtype=torch.bool, device="cuda")
    bad[20:45], bad[200:231] = True, True

    def run(qkv, dao):
        ao, lse, dqkv = torch.empty(rows, C, device="cuda"), torch.empty(H, rows, device="cuda"), torch.empty(rows, 3 * C, device="cuda")
        L.spa_packed_attention_fwd(p, qkv, seg, len(cuts) - 1, ao, lse)
        L.spa_packed_attention_bwd(p, qkv, ao, lse, dao, seg, len(cuts) - 1, dqkv)
        return ao[~bad], lse[:, ~bad], dqkv[~bad]

    want = run(qkv, dao)
    assert all(bool(torch.isfinite(w).all()) for w in want)
    for what in range(4):                              # in Q, K, V or dO
        q2, d2 = qkv.clone(), dao.clone()
        part = d2 if what == 3 else q2[:, what * C:(what + 1) * C]
        part[bad] = torch.where(rnd(int(bad.sum()), C) > 0.5, value, part[bad])
        for got, ref in zip(run(q2, d2), want):
            assert torch.allclose(got, ref, rtol=1e-5, atol=1e-5)      # sums of up to 150 terms in another order


# capacities at which one group of threads takes all streamed tiles of a CTA: segments of at most 64 rows, and any
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d,H,cap,lengths", [
    (32, 8, 3560, [49] * 30 + [1, 64, 63, 15, 17, 31, 33] + [64] * 20),
    (64, 8, 5950, [64, 49, 1] * 24 + [33] * 25),
    (32, 8, 7120, [1, 700, 64, 65, 31, 129, 32, 400] + [0] * 6),
    (64, 8, 7120, [63, 1, 333, 128, 500, 2] * 3),
])
def test_one_group_of_threads_per_cta(d, H, cap, lengths, dtype):
    from paper_2410_23608_b200 import binding as L
    C, Np, n_seg = H * d, sum(lengths), len(lengths)
    T = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(Np)
    qkv, dao = (torch.randn(cap, n * C, generator=g, device="cuda").to(T) for n in (3, 1))
    qkv[Np:], dao[Np:] = float("nan"), float("nan")    # rows past the last packed one are unspecified
    p = L.make_params(1, cap, C, H, dtype, cap, L.SPA_FLAG_SIMT_ONLY if dtype == "bf16" else 0)
    n_seg = max(n_seg, -(-cap // 64)) if max(lengths) <= 64 else n_seg        # the others are empty
    cuts = torch.tensor([0] + lengths + [0] * (n_seg - len(lengths)), device="cuda").cumsum(0).int()

    def run(qkv, dao):
        ao, lse, dqkv = (torch.full(s, 7.0, device="cuda", dtype=t) for s, t in (((cap, C), T), ((H, cap), torch.float32), ((cap, 3 * C), T)))
        L.spa_packed_attention_fwd(p, qkv, cuts, n_seg, ao, lse)
        L.spa_packed_attention_bwd(p, qkv, ao, lse, dao, cuts, n_seg, dqkv)
        return ao, lse, dqkv

    ao, lse, dqkv = run(qkv, dao)
    assert bool((ao[Np:] == 7).all()) and bool((lse[:, Np:] == 7).all()) and bool((dqkv[Np:] == 7).all())
    # fp64; sums of up to 700 terms in another order, or results and the D_i's outputs rounded to 8 bits
    rel = 1e-5 if dtype == "f32" else 1e-2
    for a, b in zip(cuts[:-1].tolist(), cuts[1:].tolist()):
        if a == b:
            continue
        x = qkv[a:b].double().view(b - a, 3, H, d).permute(1, 2, 0, 3).contiguous().requires_grad_()
        s = x[0] @ x[1].transpose(-1, -2) * d ** -0.5
        o = s.softmax(-1) @ x[2]
        o.backward(dao[a:b].double().view(b - a, H, d).transpose(0, 1))
        for got, want in ((ao[a:b], o.transpose(0, 1).reshape(b - a, C)), (lse[:, a:b], s.logsumexp(-1)),
                          (dqkv[a:b, 2 * C:], x.grad[2].transpose(0, 1).reshape(b - a, C)),
                          # those of Q and K vanish with one row: against the size of the terms
                          (dqkv[a:b, :2 * C], x.grad[:2].permute(2, 0, 1, 3).reshape(b - a, 2 * C))):
            scale = want.norm().clamp_min(0.1 * want.numel() ** 0.5)
            assert float((got.double() - want).norm()) <= rel * float(scale)
    # what the fourth segment holds stays there
    a, b = cuts[3].item(), cuts[4].item()
    q2 = qkv.clone()
    q2[a:b] = float("inf")
    keep = torch.arange(cap, device="cuda")
    keep = keep[((keep < a) | (keep >= b)) & (keep < Np)]
    for got, want in zip(run(q2, dao), (ao, lse, dqkv)):
        got, want = (got[:, keep], want[:, keep]) if got.shape[0] == H else (got[keep], want[keep])
        assert torch.allclose(got.float(), want.float(), rtol=rel, atol=rel)
