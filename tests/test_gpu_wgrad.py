"""bf16 weight gradients with their bias gradient: CTA pairs with split K, and clusters that add their partial tiles, at the
edges of tiles, 64-row blocks and splits; the input gradient beside them on pairs."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cap,n_in,n_out", [
    (0, 64, 64, 64),             # nothing selected
    (1, 1, 64, 72),              # one row
    (63, 500, 136, 64), (64, 64, 128, 128), (65, 65, 72, 200),   # around a 64-row block; remainders of a tile
    (1000, 4000, 384, 1152),     # clusters, several blocks per CTA
    (129, 8192, 520, 776),       # pairs with fewer blocks than splits, remainders of 256
    (8192, 8192, 768, 768), (9001, 18432, 768, 2304),
])
def test_weight_and_bias_gradient(rows, cap, n_in, n_out):
    from paper_2410_23608_b200 import binding as L
    g = torch.Generator(device="cuda").manual_seed(rows + n_out)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    p = L.make_params(1, cap, 64, 2, "bf16", cap)
    cu = torch.tensor([0, rows], dtype=torch.int32, device="cuda")
    a, W, dout = rnd(cap, n_in), rnd(n_out, n_in), rnd(cap, n_out)
    a[rows:], dout[rows:] = float("nan"), float("nan")      # rows past the last packed one are unspecified
    ws, status = torch.empty(160 << 20, dtype=torch.uint8, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    A, D = a[:rows].double(), dout[:rows].double()
    runs = []
    for with_da in (True, False, False):
        da = torch.full((cap, n_in), 7.0, device="cuda").bfloat16() if with_da else None
        dW, db = (torch.full(s, float("nan"), device="cuda") for s in ((n_out, n_in), (n_out,)))
        L.spa_packed_linear_bwd(p, a, W, dout, n_in, n_out, cu, da, dW, db, ws, d_status=status)
        assert L.spa_read_status(status) == 0
        for got, ref, scale in ((dW, D.T @ A, D.abs().T @ A.abs()), (db, D.sum(0), D.abs().sum(0))):
            assert bool(((got.double() - ref).abs() <= 1e-5 * scale + 1e-6).all())
        if with_da:
            ref = D @ W.double()
            assert rows == 0 or float(((da[:rows].double() - ref).abs() / (1e-2 * ref.abs() + 1e-2 * ref.abs().mean())).max()) < 1
            assert bool((da[rows:] == 7).all())
        runs.append((dW, db))
    assert torch.equal(runs[1][0], runs[2][0]) and torch.equal(runs[1][1], runs[2][1])   # bitwise reproducible
