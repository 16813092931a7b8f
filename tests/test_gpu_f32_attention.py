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
