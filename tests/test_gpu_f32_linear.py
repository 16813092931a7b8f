"""fp32 linear layers on the tensor cores (three bf16 parts per value) at the edges of their tiles and splits."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cap,n_in,n_out", [
    (1, 1, 4, 4),            # one row, layers narrower than any tile
    (127, 300, 60, 68),      # half-filled 16-byte chunks at the end of K and N
    (129, 129, 64, 132),     # one row and one column group past a tile
    (0, 64, 96, 96),         # nothing selected
    (1000, 2048, 388, 260),  # K and N that no block divides, K split over a cluster
    (2500, 2500, 96, 288),
])
def test_f32_linear_forward_and_gradients(rows, cap, n_in, n_out):
    from paper_2410_23608_b200 import binding as L
    g = torch.Generator(device="cuda").manual_seed(rows + n_in)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    p = L.make_params(1, cap, 64, 2, "f32", cap)
    cu = torch.tensor([0, rows], dtype=torch.int32, device="cuda")
    a, W, b, dout = rnd(cap, n_in), rnd(n_out, n_in), rnd(n_out), rnd(cap, n_out)
    a[rows:], dout[rows:] = float("nan"), float("nan")      # rows past the last packed one are unspecified
    out, da = torch.full((cap, n_out), 7.0, device="cuda"), torch.full((cap, n_in), 7.0, device="cuda")
    dW, db, status = torch.empty(n_out, n_in, device="cuda"), torch.empty(n_out, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    L.spa_packed_linear(p, a, W, b, n_in, n_out, cu, out, d_status=status)
    L.spa_packed_linear_bwd(p, a, W, dout, n_in, n_out, cu, da, dW, db, d_status=status)
    assert L.spa_read_status(status) == 0
    A, D = a[:rows].double(), dout[:rows].double()
    for got, ref, scale in ((out[:rows], A @ W.double().T + b.double(), A.abs() @ W.double().abs().T),
                            (da[:rows], D @ W.double(), D.abs() @ W.double().abs()),
                            (dW, D.T @ A, D.abs().T @ A.abs()), (db, D.sum(0), D.abs().sum(0))):
        # the bound of an fp32 sum: a few roundings of the sum of magnitudes
        assert bool(((got.double() - ref).abs() <= 2e-6 * scale + 1e-6).all())
    assert bool((out[rows:] == 7.0).all()) and bool((da[rows:] == 7.0).all())


@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("rows,cap,n_in,n_out", [(129, 129, 64, 132), (1000, 2048, 388, 260)])   # one CTA per tile; K split over a cluster
def test_f32_linear_keeps_infinities(rows, cap, n_in, n_out, large):
    """Infinite operands, and finite ones that round to infinity in bf16 (above 3.39e38), give what a chain of fp32 FMAs
    gives: infinities of the right sign, NaN only where the sum has it, everything else untouched."""
    from paper_2410_23608_b200 import binding as L
    g = torch.Generator(device="cuda").manual_seed(rows)
    # multiples of 1/16 up to 1/2 in size: their second and third bf16 parts are zero, and so are some of the values
    rnd = lambda *s: torch.randint(-8, 9, s, generator=g, device="cuda").float() / 16
    p = L.make_params(1, cap, 64, 2, "f32", cap)
    cu = torch.tensor([0, rows], dtype=torch.int32, device="cuda")
    a, W, dout = rnd(cap, n_in), rnd(n_out, n_in), rnd(cap, n_out)
    if large:
        a[90, 31], dout[91, 33], W[50, 34] = 3.4e38, -3.4e38, 3.4e38
    else:
        a[3, 5], a[7, 0], a[7, 63], a[20, 9] = float("inf"), float("inf"), float("-inf"), float("nan")
        dout[4, 2], dout[40, 11], W[17, 30], W[60, 1] = float("-inf"), float("inf"), float("inf"), float("-inf")
    out, da = torch.empty(cap, n_out, device="cuda"), torch.empty(cap, n_in, device="cuda")
    dW, db, status = torch.empty(n_out, n_in, device="cuda"), torch.empty(n_out, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    L.spa_packed_linear(p, a, W, None, n_in, n_out, cu, out, d_status=status)
    L.spa_packed_linear_bwd(p, a, W, dout, n_in, n_out, cu, da, dW, db, d_status=status)
    assert L.spa_read_status(status) == 0
    A, D, W64, one = a[:rows].double(), dout[:rows].double(), W.double(), torch.ones(rows, 1, device="cuda").double()
    finite = lambda t: torch.nan_to_num(t, 0.0, 0.0, 0.0)
    infinities = 0
    for got, x, y in ((out[:rows], A, W64.T), (da[:rows], D, W64), (dW, D.T, A), (db[:, None], D.T, one)):
        # x @ y in fp64, with the terms that hold an infinity or NaN looked at one by one
        ref = finite(x) @ finite(y)
        for k in torch.nonzero(~(torch.isfinite(x).all(0) & torch.isfinite(y).all(1)))[:, 0].tolist():
            ref += x[:, k, None] * y[None, k] - finite(x[:, k, None]) * finite(y[None, k])
        got = got.double()
        assert torch.equal(torch.isnan(got), torch.isnan(ref)) and torch.equal(got[torch.isinf(ref)], ref[torch.isinf(ref)])
        infinities += int(torch.isinf(ref).sum())
        ok = torch.isfinite(ref)
        # the bound of an fp32 sum: a few roundings of the sum of magnitudes
        assert bool(((got - ref).abs() <= 2e-6 * (finite(x).abs() @ finite(y).abs()) + 1e-6)[ok].all())
    assert large == (infinities == 0)
