"""A training step of the block as one CUDA graph: no kernel of it waits for two others, which would cost it its early launch."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


def edges(graph):
    """(from, to) node handles of a captured graph."""
    rt = ctypes.CDLL("libcudart.so.12")
    n = ctypes.c_size_t(0)
    h = ctypes.c_void_p(graph.raw_cuda_graph())
    assert rt.cudaGraphGetEdges_v2(h, None, None, None, ctypes.byref(n)) == 0
    a, b, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (ctypes.c_uint64 * n.value)()
    assert rt.cudaGraphGetEdges_v2(h, a, b, data, ctypes.byref(n)) == 0
    return list(zip(a, b))


@pytest.mark.parametrize("dtype,C,H", [("bf16", 384, 6), ("bf16", 768, 12)])
@pytest.mark.parametrize("trainable", [False, True])
def test_every_kernel_of_a_step_has_one_predecessor(dtype, C, H, trainable):
    from paper_2410_23608_b200 import binding as L
    from paper_2410_23608_b200.block import SpaBlock
    B, N = 24, 196
    rnd = lambda *s, std=1.0: (torch.randn(*s, device="cuda") * std).to(torch.bfloat16)
    x, dY, w_g = rnd(B, N, C), rnd(B, N, C), rnd(C, std=C ** -0.5)
    W = (rnd(3 * C, C, std=C ** -0.5), rnd(3 * C), rnd(C, C, std=C ** -0.5), rnd(C))
    labels = torch.ones(B * N, dtype=torch.uint8, device="cuda")
    blk = SpaBlock(B, N, C, H, dtype, flags=L.SPA_FLAG_GATE_SCALE | L.SPA_FLAG_RESIDUAL if trainable else 0)

    def step():
        blk.forward(x, w_g, 0.0, *W)
        if trainable:
            blk.backward_trainable(dY, x, w_g, labels=labels)
        else:
            blk.backward(dY)

    names = ("dX", "dW_qkv", "db_qkv", "dW_o", "db_o") + (("dw_g", "db_g") if trainable else ())
    step()
    torch.cuda.synchronize()
    want = [getattr(blk, k).clone() for k in names]
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        step()
    into = [b for _, b in edges(g)]
    assert len(into) >= 10 and len(into) == len(set(into))
    g.instantiate()
    for _ in range(3):
        for k in names:
            getattr(blk, k).zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(getattr(blk, k), w) for k, w in zip(names, want))
    assert blk.read_status() == 0
