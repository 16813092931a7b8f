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
