"""The transformer block as one call on each of its kernel paths, against the fp64 oracle: fused epilogues (single CTAs; CTA
pairs are in test_gpu_layer.py), calls of their own on the fp32-FMA path, separate scatter kernels."""
import numpy as np
import pytest
import torch

from oracle import spa_oracle as O
from tests.gpu_util import assert_close, dev, host
from tests.test_gpu_layer import layer_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flag", ["SPA_FLAG_SIMT_ONLY", "SPA_FLAG_UNFUSED", "SPA_FLAG_NO_CTA_PAIRS"])
@pytest.mark.parametrize("ci,B", [(1, 1), (2, 1)])
def test_layer_paths(ci, B, flag):
    from paper_2410_23608_b200 import binding as L
    from paper_2410_23608_b200.layer import SpaLayer
    cfg, inp, x, prm, f = layer_problem(ci, B)
    bwd = O.layer_bwd(f, inp.dY, x, prm, cfg.H)
    dt = cfg.dtype
    dprm = {k: (dev(v, dt) if isinstance(v, np.ndarray) else v) for k, v in prm.items()}
    lay = SpaLayer(cfg.B, cfg.N, cfg.C, cfg.H, dt, flags=getattr(L, flag))
    for _ in range(2):
        out = lay.forward(dev(x, dt), dprm)
        dX = lay.backward(dev(inp.dY, dt))
    torch.cuda.synchronize()
    assert lay.read_status() == 0
    assert np.array_equal(lay.blk.mask.cpu().numpy().astype(bool), f["spa"]["mask"].reshape(-1))
    for name, got, ref in (("out", out, f["out"]), ("h", lay.h, f["h"]), ("dX", dX, bwd["dX"]), ("dW1", lay.dW1, bwd["dW1"]),
                           ("db1", lay.db1, bwd["db1"]), ("dg1", lay.dg1, bwd["dg1"]), ("dbe2", lay.dbe2, bwd["dbe2"]),
                           ("dW_qkv", lay.blk.dW_qkv, bwd["dW_qkv"])):
        assert_close(host(got), ref, dt, name, scale_max_abs=True)


# rows around the line between narrow and wide tiles of the single-CTA products (148 wide tiles), remainders of both
@pytest.mark.parametrize("rows,n_in,n_out", [(1, 64, 72), (129, 136, 64), (2368, 72, 1024), (2369, 64, 1024), (2432, 64, 1032),
                                             (6272, 384, 384), (18944, 64, 128), (18945, 64, 120)])
@pytest.mark.parametrize("slack", [0, 300, 20000])   # capacity past the rows: narrow tiles, chosen by the rows, wide
def test_linear_tile_widths(rows, n_in, n_out, slack):
    from paper_2410_23608_b200 import binding as L
    g = torch.Generator(device="cuda").manual_seed(rows)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    cap = rows + slack
    p = L.make_params(1, cap, 64, 2, "bf16", cap, flags=L.SPA_FLAG_NO_CTA_PAIRS)
    cu = torch.tensor([0, rows], dtype=torch.int32, device="cuda")
    a, W, b, dout = rnd(cap, n_in), rnd(n_out, n_in), rnd(n_out), rnd(cap, n_out)
    a[rows:], dout[rows:] = float("nan"), float("nan")
    out, da = torch.full((cap, n_out), 7.0, device="cuda").bfloat16(), torch.full((cap, n_in), 7.0, device="cuda").bfloat16()
    ws, status = torch.empty(64 << 20, dtype=torch.uint8, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    L.spa_packed_linear(p, a, W, b, n_in, n_out, cu, out, d_status=status)
    L.spa_packed_linear_bwd(p, a, W, dout, n_in, n_out, cu, da, None, None, ws, d_status=status)
    assert L.spa_read_status(status) == 0
    for got, ref in ((out[:rows], a[:rows].double() @ W.double().T + b.double()), (da[:rows], dout[:rows].double() @ W.double())):
        assert float(((got.double() - ref).abs() / (1e-2 * ref.abs() + 1e-2 * ref.abs().mean())).max()) < 1
    assert bool((out[rows:] == 7).all()) and bool((da[rows:] == 7).all())


def test_inplace_flag_changes_nothing():
    from paper_2410_23608_b200 import binding as L
    from paper_2410_23608_b200.layer import SpaLayer
    cfg, inp, x, prm, _ = layer_problem(2, 1)
    dprm = {k: (dev(v, cfg.dtype) if isinstance(v, np.ndarray) else v) for k, v in prm.items()}
    runs = []
    for flags in (0, L.SPA_FLAG_INPLACE):
        lay = SpaLayer(cfg.B, cfg.N, cfg.C, cfg.H, cfg.dtype, flags=flags)
        xd = dev(x, cfg.dtype)
        out, dX = lay.forward(xd, dprm), lay.backward(dev(inp.dY, cfg.dtype))
        torch.cuda.synchronize()
        assert lay.read_status() == 0 and torch.equal(xd, dev(x, cfg.dtype))
        runs.append((out, dX, lay.dW1, lay.blk.dW_qkv))
    assert all(torch.equal(a, b) for a, b in zip(*runs))


def test_activation_of_the_product_is_that_of_the_call_within_a_rounding():
    from paper_2410_23608_b200 import binding as L
    from paper_2410_23608_b200.layer import SpaLayer
    cfg, inp, x, prm, _ = layer_problem(2, 2)
    dprm = {k: (dev(v, cfg.dtype) if isinstance(v, np.ndarray) else v) for k, v in prm.items()}
    lay = SpaLayer(cfg.B, cfg.N, cfg.C, cfg.H, cfg.dtype)
    lay.forward(dev(x, cfg.dtype), dprm)
    by_call = torch.empty_like(lay.h)
    L.spa_gelu(lay.p, lay.u, lay.hidden, by_call)
    exact = torch.nn.functional.gelu(lay.u.double())
    for h in (lay.h.double(), by_call.double()):
        # the rounding to eight bits (at most 2^-8 of the value), and the error of the distribution function times |u|
        assert bool(((h - exact).abs() <= 2.0 ** -8 * exact.abs() + 6e-7 * lay.u.double().abs() + 1e-30).all())
    assert float((lay.h != by_call).double().mean()) < 2e-3
